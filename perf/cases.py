"""Performance cases: what a user of this package has it do, through its public entry points.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)`` one more of the
same ranges; ``prepare(case, seed)`` makes what the program holds before the call (input particles
on the GPU, species stores, tables), ``run(state)`` is one pass, ``work(case)`` the bytes and
operations the pass cannot do without, and ``exact(case, seed)`` the same outputs in 64 bits from
plain torch and numpy.

Kinds of case:
  steps   copy a population in, take ``steps`` steps with one ``qed.run``, read counts and ledger
  job     a whole head-on collision: electrons in, optical depths drawn, ``qed.run_multistep``
  pic     a PIC code's time loop: one ``qed.run`` of one step per call, fields gathered from a grid
  batch   a parameter scan: scenarios attached to a ``qed.Batch`` and advanced together
  merge   macroparticle merging of a photon population
  noalloc the allocation-free emission step on the caller's own arrays, in a time loop

Units: momenta in m c, fields in the Schwinger field, time in hbar/(m c^2), length in hbar/(m c).
"""
import math

import numpy as np
import torch

from paper_1311_5551_gb300 import qed

TIME_S = 1.0545718176461565e-34 / (9.1093837015e-31 * 299792458.0 ** 2)  # s per hbar/(m c^2)
LENGTH_M = TIME_S * 299792458.0                                          # m per hbar/(m c)
ALPHA = 7.2973525693e-3

_COLS = ("x", "y", "z", "ux", "uy", "uz")


# ------------------------------------------------------------------------------------- the cases
def listed():
    return [
        # test problem 1 (uniform B, eta0 = 1, photons drained) at the smallest size in use: each
        # step is a few microseconds of work, so launches and latency count
        dict(name="uniform_b_1e3", kind="steps", field="uniform", prec="mixed", n_e=1000, n_p=0, n_g=0, steps=200,
             gamma=1000.0, strength=1e-3, pairs=False, drain=True, recoil=False),
        # the same problem on the FP64 path, at the size the paper's checks use (an odd number)
        dict(name="uniform_b_fp64_1e4", kind="steps", field="uniform", prec="fp64", n_e=10007, n_p=0, n_g=0, steps=100,
             gamma=1000.0, strength=1e-3, pairs=False, drain=True, recoil=False),
        # test problem 2 (circularly polarised wave, gamma0 = 4120) on the FP64 path, whole: 20 steps
        dict(name="cp_wave_fp64_1e5", kind="steps", field="cp", prec="fp64", n_e=100000, n_p=0, n_g=0, steps=20,
             gamma=4120.0, strength=1.22e-4, pairs=True, drain=False, recoil=False),
        # a small collision of the scan, whole (4000 steps, event-free stretches taken in one pass)
        dict(name="collision_1e3", kind="job", n_e=1000, a0=250.0, gamma=2000.0, fwhm_fs=30.0, steps=4000, chunk=64),
        # the head-on collision of the benchmark, whole: 1e6 electrons, a0 = 100, 4000 steps
        dict(name="collision_1e6", kind="job", n_e=1000000, a0=100.0, gamma=2000.0, fwhm_fs=30.0, steps=4000, chunk=64),
        # the densest part of a collision: a bunch in the pulse with the photons it has made so far
        dict(name="in_pulse_3e5", kind="steps", field="lp", prec="mixed", n_e=300000, n_p=300, n_g=6000000, steps=64,
             gamma=2000.0, strength=100.0, pairs=True, drain=False, recoil=False),
        # strong pulse, many pairs: a0 = 400, gamma = 4000, energy-conserving recoil
        dict(name="pair_rich_2e4", kind="steps", field="lp", prec="mixed", n_e=20000, n_p=5000, n_g=500001, steps=200,
             gamma=4000.0, strength=400.0, pairs=True, drain=False, recoil=True),
        # the rotating-field cascade late in its run: few leptons among many photons
        dict(name="cascade_2e7", kind="steps", field="rotating", prec="mixed", n_e=20000, n_p=10000, n_g=20000000,
             steps=50, gamma=400.0, strength=1e-3, pairs=True, drain=False, recoil=False),
        # a PIC code's loop: one step per call, fields from its grid (linear weights)
        dict(name="pic_cic_2e5", kind="pic", prec="mixed", shape=1, n_e=200003, n_p=0, n_g=200000, steps=16, cells=48,
             gamma=1000.0),
        # merging the photons of a cascade (bench's bins: 8^3 cells, 6 x 6 per cube face, 2 per octave)
        dict(name="merge_3e6", kind="merge", prec="mixed", n=3000000, cells=8, n_face=6, n_sub=2, min_group=4),
        # a parameter scan in a batch: 24 collisions of 1e3..2e5 electrons, 256 steps in the pulse
        dict(name="scan_24", kind="batch", slots=24, n_min=1000, n_max=200000, steps=256),
        # the allocation-free step in a host code's time loop
        dict(name="noalloc_3e4", kind="noalloc", prec="mixed", n=30000, steps=8, gamma=1000.0, strength=1e-3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "job", "pic", "merge", "batch", "noalloc"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    if kind == "steps":
        field = rng.choice(["uniform", "lp", "cp", "rotating"])
        small = prec == "fp64"  # the FP64 path is about ten times slower per particle
        n_e = _log_int(rng, 100, 30000 if small else 300000)
        n_g = 0 if field == "uniform" else _log_int(rng, 100, 300000 if small else 10000000)
        drain = field == "uniform" and rng.random() < 0.7
        gamma = rng.uniform(200.0, 4000.0)
        strength = {"uniform": 1.0 / gamma, "lp": rng.uniform(10.0, 500.0), "cp": 1.22e-4,
                    "rotating": 1e-3}[field]
        return dict(kind="steps", field=field, prec=prec, n_e=n_e, n_p=_log_int(rng, 1, max(2, n_e // 4)), n_g=n_g,
                    steps=_log_int(rng, 1, 100), gamma=gamma, strength=strength, pairs=rng.random() < 0.8, drain=drain,
                    recoil=rng.random() < 0.3)
    if kind == "job":
        a0 = rng.uniform(10.0, 500.0)
        return dict(kind="job", n_e=_log_int(rng, 1000, min(3e5, 2e7 / a0)), a0=a0, gamma=rng.uniform(200.0, 4000.0),
                    fwhm_fs=rng.uniform(15.0, 45.0), steps=rng.randint(2000, 4000), chunk=rng.choice([16, 64]))
    if kind == "pic":
        return dict(kind="pic", prec=prec, shape=rng.choice([1, 2]), n_e=_log_int(rng, 1000, 200000),
                    n_p=rng.randint(0, 2000), n_g=_log_int(rng, 1000, 300000), steps=rng.randint(1, 16),
                    cells=rng.randint(8, 64), gamma=rng.uniform(200.0, 2000.0))
    if kind == "merge":
        return dict(kind="merge", prec=prec, n=_log_int(rng, 1000, 10000000), cells=rng.choice([4, 8, 16]),
                    n_face=rng.choice([6, 8]), n_sub=rng.choice([1, 2, 4]), min_group=rng.randint(3, 6))
    if kind == "batch":
        return dict(kind="batch", slots=rng.randint(2, 24), n_min=1000, n_max=_log_int(rng, 2000, 200000),
                    steps=rng.randint(40, 256))
    return dict(kind="noalloc", prec=prec, n=_log_int(rng, 100, 65536), steps=rng.randint(1, 16),
                gamma=rng.uniform(200.0, 2000.0), strength=1e-3)


# ------------------------------------------------------------------------------------- inputs
def _omega(lam_m):
    return 2.0 * math.pi * LENGTH_M / lam_m


def _pulse(a0, gamma, fwhm_fs, meet):
    """Linearly polarised pulse along +x (lambda = 1 um, sin^2 envelope) whose centre meets the
    bunch at step ``meet``; dt = lambda/(100 c); the window moves with the bunch along -x."""
    om = _omega(1e-6)
    dt = 2.0 * math.pi / om / 100.0
    length = fwhm_fs * 1e-15 / (1.0 - 2.0 * math.asin(2.0 ** -0.25) / math.pi) / TIME_S
    beta = math.sqrt(1.0 - 1.0 / gamma ** 2)
    fld = dict(kind=qed.FIELD_PLANE_LP, E0=a0 * om, omega=om, phi_start=om * meet * dt - 0.5 * om * length,
               phi_len=om * length)
    return fld, dt, beta * meet * dt, -1.0


def _setting(case):
    """Field, time step, first step and window of a 'steps' case."""
    f = case["field"]
    if f == "uniform":
        cb = case["strength"]
        gyro = 2.0 * math.pi * case["gamma"] / cb
        return dict(kind=qed.FIELD_UNIFORM, B=(0.0, 0.0, cb)), gyro / 1000.0, 0, 0.0, 0.0
    if f == "lp":
        fld, dt, x0, v = _pulse(case["strength"], case["gamma"], 30.0, 2000)
        return fld, dt, 2000 - case["steps"] // 2, x0, v
    if f == "cp":
        e0 = case["strength"]
        dt_qed = math.pi / (math.sqrt(3.0) * ALPHA * e0 * 5.0 * math.pi / 3.0)
        return dict(kind=qed.FIELD_PLANE_CP, E0=e0, omega=_omega(1e-6)), 0.3 * dt_qed, 0, 0.0, 0.0
    om = _omega(0.8e-6)
    return dict(kind=qed.FIELD_ROTATING_E, E0=case["strength"], omega=om), 2.0 * math.pi / om / 200.0, 1000, 0.0, 0.0


def _real(case):
    return torch.float64 if case.get("prec") == "fp64" else torch.float32


def _directions(g, n, spread, planar):
    """Unit vectors: along -x with a small spread (a beam), or in the plane of a rotating field."""
    if planar:
        ph = 2.0 * math.pi * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
        z = 0.05 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
        d = torch.stack([torch.cos(ph), torch.sin(ph), z])
    else:
        t = spread * torch.randn((2, n), generator=g, device="cuda", dtype=torch.float64)
        d = torch.stack([-torch.ones(n, device="cuda", dtype=torch.float64), t[0], t[1]])
    return d / d.norm(dim=0)


def _population(g, n, kind, gamma, spread, planar, size, real, mono=False):
    """Columns x, y, z, ux, uy, uz (species precision) and the FP64 optical depths of n particles:
    leptons of about gamma m c^2 (5% rms), photons with the soft synchrotron spectrum
    eps^(-2/3) up to gamma/2."""
    d = _directions(g, n, spread, planar)
    if kind == qed.PHOTON:
        e = (0.5 * gamma - 1e-3) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64) ** 3 + 1e-3
        u = d * e
    else:
        gam = torch.full((n,), gamma, device="cuda", dtype=torch.float64)
        if not mono:
            gam = (gam * (1.0 + 0.05 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64))).clamp(min=1.5)
        u = d * torch.sqrt(gam * gam - 1.0)
    x = size * torch.randn((3, n), generator=g, device="cuda", dtype=torch.float64)
    tau = -torch.log1p(-torch.rand(n, generator=g, device="cuda", dtype=torch.float64)).clamp(max=-1e-12)
    return [c.to(real).contiguous() for c in (*x, *u)] + [tau]


def _inputs(case, seed):
    """Input particles per species (e-, e+, photons) of a 'steps', 'pic', 'job' or 'noalloc' case."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    real = _real(case)
    um = 1e-6 / LENGTH_M
    f = case.get("field", {"job": "lp", "pic": "grid"}.get(case["kind"], "uniform"))
    planar = f in ("rotating", "grid")
    size = {"uniform": 0.0, "cp": 0.0, "grid": 1.0, "rotating": 2.0 * um}.get(f, 1.0 * um)
    spread = {"uniform": 0.0, "cp": 0.0}.get(f, 1e-3)
    ns = (case.get("n_e", case.get("n")), case.get("n_p", 0), case.get("n_g", 0))
    out = []
    for kind, n in zip((qed.ELECTRON, qed.POSITRON, qed.PHOTON), ns):
        wide = 0.05 if kind != qed.ELECTRON and f == "lp" else spread  # photons and e+ leave at about a0/gamma
        out.append(_population(g, n, kind, case["gamma"], wide, planar, size, real, mono=f in ("uniform", "cp")))
    if f == "uniform":  # test problem 1: all electrons along x, perpendicular to B
        for cols in out[:2]:
            cols[3].neg_()
    if f == "grid":  # spread over the box
        for cols in out:
            for c in range(3):
                cols[c] = ((torch.rand(cols[c].shape, generator=g, device="cuda", dtype=torch.float64) - 0.5)
                           * _BOX).to(real)
    return out


_BOX = 3.2e6  # side of the grid's box (holds the orbits of test problem 1)


def _grid_field(case, seed):
    """A PIC grid: cB_z = 1e-3 with a 10% random perturbation of every component."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    n = case["cells"]
    a = 1e-4 * torch.randn((6, n - 3, n - 1, n), generator=g, device="cuda", dtype=torch.float32)
    a[5] += 1e-3
    spc = tuple(_BOX / (m - 1) for m in (n, n - 1, n - 3))
    return a.to(_real(case)).contiguous(), (-0.5 * _BOX,) * 3, spc


def _merge_inputs(case, seed):
    """Photons of a cascade: emitted over a long run in the plane of the field, flying outward."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n, real = case["n"], _real(case)
    cols = _population(g, n, qed.PHOTON, 400.0, 0.0, True, 0.0, torch.float64)
    r = 2.0e7 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    k = torch.stack(cols[3:6])
    x = r * k / k.norm(dim=0) + 1e6 * torch.randn((3, n), generator=g, device="cuda", dtype=torch.float64)
    return [c.to(real).contiguous() for c in (*x, *cols[3:6])] + [cols[6]], 2.3e7


# ------------------------------------------------------------------------------------- prepare
_TABLES = []


def _tables():
    if not _TABLES:
        _TABLES.append(qed.Tables())
    return _TABLES[0]


class _Array:
    """A device array of a species, seen by torch (and keeping the species alive)."""

    def __init__(self, species, ptr, n, typestr):
        self.species = species
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (n,), "typestr": typestr, "version": 3}


def _columns(sp):
    """The species' own device arrays as tensors (mixed path: the optical depth's two floats)."""
    v = sp.view()
    real = "<f4" if sp.precision == qed.MIXED else "<f8"
    out = {k: torch.as_tensor(_Array(sp, getattr(v.arrays, k), sp.capacity, real), device="cuda") for k in _COLS}
    if sp.precision == qed.MIXED:
        pair = torch.as_tensor(_Array(sp, v.arrays.tau, 2 * sp.capacity, "<f4"), device="cuda").view(-1, 2)
        out["tau"], out["tau_low"] = pair[:, 0], pair[:, 1]
    else:
        out["tau"] = torch.as_tensor(_Array(sp, v.arrays.tau, sp.capacity, "<f8"), device="cuda")
    out["id"] = torch.as_tensor(_Array(sp, v.arrays.id, sp.capacity, "<i4"), device="cuda")
    return out


def _soa(cols):
    return qed.Soa(*[c.data_ptr() for c in cols[:6]], cols[6].data_ptr() if len(cols) > 6 else None, None)


def _load(sp, cols):
    n = cols[0].numel() if cols else 0
    sp.upload_soa(_soa(cols) if n else qed.Soa(*([None] * 8)), n, n)


def _caps(n, a0, gamma, fwhm_fs):
    dur = 0.5 + 0.5 * fwhm_fs / 30.0
    pairs = int(n * 2.5 * (gamma * a0 / 1e6) ** 1.2 * dur) + 4096
    return n + pairs, pairs, int(n * (a0 * dur * (0.5 + 0.25 * gamma / 1000.0) + 16)) + 4096


def _stores(prec, e_cap, p_cap, g_cap, d_cap=0):
    sp = [qed.Species(qed.ELECTRON, prec, e_cap, p_cap), qed.Species(qed.POSITRON, prec, p_cap, p_cap),
          qed.Species(qed.PHOTON, prec, g_cap, e_cap + p_cap)]
    return sp + ([qed.Species(qed.PHOTON, prec, d_cap, 1)] if d_cap else [])


def _step_caps(case):
    """Room for a few events per lepton (and for the pairs of the strongest fields)."""
    lep = case["n_e"] + case["n_p"]
    made = int(1.2 * lep * min(case["steps"], 40 + case["steps"] // 2)) + 4096
    pairs = case["n_g"] // 2 + lep + 65536 if case.get("pairs", True) else 4096
    return case["n_e"] + pairs, case["n_p"] + pairs, case["n_g"] + made + 4 * pairs


def prepare(case, seed):
    kind = case["kind"]
    prec = qed.FP64 if case.get("prec") == "fp64" else qed.MIXED
    s = {"case": case, "kind": kind, "tables": _tables(), "seed": int(seed)}
    if kind in ("steps", "pic"):
        s["in"] = _inputs(case, seed)
        if kind == "steps":
            fld, dt, s["first"], x0, v = _setting(case)
            opt = dict(make_pairs=case["pairs"], drain_photons=case["drain"], recoil_energy=case["recoil"])
        else:
            grid, org, spc = _grid_field(case, seed)
            fld = dict(kind=qed.FIELD_GRID, grid=grid, shape=case["shape"], origin=org, spacing=spc)
            dt, s["first"], x0, v, opt = 2.0 * math.pi * 1000.0 / 1e-3 / 1000.0, 0, 0.0, 0.0, {}
        e_cap, p_cap, g_cap = _step_caps(case)
        s["sp"] = _stores(prec, e_cap, p_cap, g_cap, g_cap if opt.get("drain_photons") else 0)
        s["params"] = qed.StepParams(dt=dt, seed=s["seed"], field=qed.Field(**fld), window_x0=x0, window_v=v, **opt)
        s["cols"] = [_columns(sp) for sp in s["sp"]]
    elif kind == "job":
        s["in"] = _inputs(case, seed)
        fld, dt, x0, v = _pulse(case["a0"], case["gamma"], case["fwhm_fs"], case["steps"] // 2)
        s["sp"] = _stores(prec, *_caps(case["n_e"], case["a0"], case["gamma"], case["fwhm_fs"]))
        s["params"] = qed.StepParams(dt=dt, seed=s["seed"], field=qed.Field(**fld), window_x0=x0, window_v=v)
        s["cols"] = [_columns(sp) for sp in s["sp"]]
    elif kind == "batch":
        s["slots"], s["batch"], room = [], qed.Batch(s["tables"], prec, case["slots"]), [0, 0, 0]
        lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
        for k in range(case["slots"]):
            # sizes, a0 and gamma spread evenly over their ranges, so that the work does not depend on the seed
            n = int(round(math.exp(lo + (hi - lo) * (k + 0.5) / case["slots"])))
            a0 = 10.0 + 490.0 * ((7 * k + 3) % case["slots"]) / case["slots"]
            gamma, fwhm = 200.0 + 3800.0 * ((5 * k + 1) % case["slots"]) / case["slots"], 30.0
            cols = _inputs(dict(kind="job", prec="mixed", n_e=n, gamma=gamma), s["seed"] + k)[0][:6]
            fld, dt, x0, v = _pulse(a0, gamma, fwhm, 2000)
            e_cap, p_cap, g_cap = _caps(n, a0, gamma, fwhm)
            sp = _stores(prec, e_cap, p_cap, min(g_cap, n * case["steps"]) + 4096)
            p = qed.StepParams(dt=dt, seed=s["seed"], scenario=k, field=qed.Field(**fld), window_x0=x0, window_v=v)
            s["slots"].append((sp, cols, p, [_columns(t) for t in sp]))
            room = [r + t.capacity for r, t in zip(room, sp)]
        s["made"] = [_result(s["slots"][0][3][j], room[j]) for j in range(3)]
    elif kind == "merge":
        cols, span = _merge_inputs(case, seed)
        s["in"] = [cols]
        s["sp"] = [qed.Species(qed.PHOTON, prec, case["n"] + 64, 64)]
        s["left"] = _result(_columns(s["sp"][0]), case["n"])
        s["bins"] = dict(origin=(-span,) * 3, cell=(2.0 * span / case["cells"],) * 3, n_cells=(case["cells"],) * 3,
                         n_face=case["n_face"], n_sub=case["n_sub"], min_group=case["min_group"])
    else:
        real = _real(case)
        n, cap = case["n"], case["n"] * case["steps"] + 64
        cols = _inputs(case, seed)[0]
        tau = cols[6]
        if prec == qed.MIXED:  # the stored form: (hi, lo) float pairs in the 8 bytes
            hi = tau.float()
            tau = torch.stack([hi, (tau - hi.double()).float()], dim=1).contiguous().view(torch.float64)[:, 0]
        s["pristine"] = [*cols[:6], tau, torch.arange(n, device="cuda", dtype=torch.int32)]
        mine = [c.clone() for c in s["pristine"]]
        names = (*_COLS, "tau", "id")
        s["e"] = dict(zip(names, mine))
        s["g"] = {k: torch.zeros(cap, device="cuda", dtype=real) for k in _COLS}
        s["g"]["tau"] = torch.zeros(cap, device="cuda", dtype=torch.float64)
        s["g"]["id"] = torch.zeros(cap, device="cuda", dtype=torch.int32)
        s["counter"] = torch.zeros(3, device="cuda", dtype=torch.int32)
        cb = case["strength"]
        s["params"] = qed.StepParams(dt=2.0 * math.pi * case["gamma"] / cb / 1000.0, seed=s["seed"],
                                     field=qed.Field(B=(0.0, 0.0, cb)))
        s["prec"] = prec
    return s


# ------------------------------------------------------------------------------------- run
def _result(cols, n):
    """Arrays of n entries for the particles a pass leaves (the rest stays zero)."""
    return {k: torch.zeros(n, device="cuda", dtype=t.dtype) for k, t in cols.items()}


def _held(cols, n_in, names):
    """The species' own arrays: the particles that went in, and the room for those made since
    (zero where nothing was made)."""
    out = {}
    for name, c, n in zip(names, cols, n_in):
        if n:
            out[name] = {k: t[:n] for k, t in c.items()}
        if n < len(c["id"]):
            out["new_" + name] = {k: t[n:] for k, t in c.items()}
    return out


def _ledger(sps):
    led = qed.read_ledger(sps)
    return np.array([*led["n"], *led["energy"], led["emitted_n"], led["emitted_energy"], led["pairs_n"],
                     led["pair_energy"]])


_NAMES = ("electrons", "positrons", "photons")


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "merge":
        sp, left = state["sp"][0], state["left"]
        _load(sp, state["in"][0])
        groups = sp.merge(**state["bins"])
        n = sp.count()
        cols = _columns(sp)
        torch._foreach_copy_([t[:n] for t in left.values()], [cols[k][:n] for k in left])
        return {"groups": groups, "count": n, "photons": left}
    if kind == "noalloc":
        torch._foreach_copy_(list(state["e"].values()), state["pristine"])
        state["counter"].zero_()
        for k in range(case["steps"]):
            qed.step_emit_noalloc(state["tables"], state["prec"], state["e"], case["n"], state["g"], state["counter"],
                                  state["params"], k)
        return {"electrons": _pairs_apart(state["e"], state["prec"]), "photons": _pairs_apart(state["g"], state["prec"]),
                "counter": state["counter"]}
    if kind == "batch":
        batch = state["batch"]
        for k, (sp, cols, params, _) in enumerate(state["slots"]):
            _load(sp[0], cols)
            sp[0].init_tau(state["seed"], k)
            _load(sp[1], None)
            _load(sp[2], None)
            batch.attach(k, sp, params, 2000 - case["steps"] // 2, case["steps"])
        batch.run(case["steps"])
        out = {"ledger": np.stack([_ledger(sp) for sp, _, _, _ in state["slots"]])}
        counts = [[t.count() for t in sp] for sp, _, _, _ in state["slots"]]
        for j, name in enumerate(_NAMES):
            made = state["made"][j]
            m = sum(c[j] for c in counts)
            for col, res in made.items():  # all scenarios' particles of a species, end to end
                torch.cat([cols[j][col][:c[j]] for (_, _, _, cols), c in zip(state["slots"], counts)], out=res[:m])
            out[name] = made
        out["counts"] = np.array(counts)
        return out
    sp, params = state["sp"], state["params"]
    if kind == "job":
        _load(sp[0], state["in"][0][:6])
        sp[0].init_tau(state["seed"])
        _load(sp[1], None)
        _load(sp[2], None)
        qed.run_multistep(state["tables"], sp, params, 0, case["steps"], case["chunk"])
        n_in = (case["n_e"], 0, 0)
    else:
        for s, cols in zip(sp, state["in"]):
            _load(s, cols)
        if len(sp) > 3:
            _load(sp[3], None)
        if kind == "steps":
            qed.run(state["tables"], sp, params, state["first"], case["steps"])
        else:
            for k in range(case["steps"]):
                qed.run(state["tables"], sp, params, state["first"] + k, 1)
        n_in = (case["n_e"], case["n_p"], case["n_g"])
    out = {"ledger": _ledger(sp), "counts": [s.count() for s in sp]}
    if case.get("drain"):  # no pairs and no photons in flight: the electrons and what they emitted
        return {**out, **_held(state["cols"][::3], (case["n_e"], 0), ("electrons", "drained"))}
    return {**out, **_held(state["cols"], n_in, _NAMES)}


def _pairs_apart(arrays, prec):
    if prec != qed.MIXED:
        return arrays
    t = arrays["tau"].view(torch.float32).view(-1, 2)
    return {**{k: v for k, v in arrays.items() if k != "tau"}, "tau": t[:, 0], "tau_low": t[:, 1]}


# ------------------------------------------------------------------------------------- work
def work(case):
    """Input particles read once, final particles written once; about 90 operations per particle
    and step for a photon in a field, 150 for an electron or positron (push, eta, rate)."""
    kind, b = case["kind"], (60 if case.get("prec") == "fp64" else 36)
    if kind == "merge":
        return {"bytes": 2.0 * b * case["n"], "flops": 40.0 * case["n"]}
    if kind == "noalloc":
        rate = 0.014 * case["gamma"] / 1000.0  # events per electron and step
        return {"bytes": b * case["n"] * (2.0 + rate * case["steps"]), "flops": 150.0 * case["n"] * case["steps"]}
    if kind == "batch":
        lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
        by = fl = 0.0
        for k in range(case["slots"]):
            n = math.exp(lo + (hi - lo) * (k + 0.5) / case["slots"])
            made = n * case["steps"] * 1.1e-3 * (10.0 + 490.0 * ((7 * k + 3) % case["slots"]) / case["slots"]) * 0.5
            by += b * (2.0 * n + made)
            fl += case["steps"] * (150.0 * n + 90.0 * 0.5 * made)
        return {"bytes": by, "flops": fl}
    if kind == "job":
        n, made = case["n_e"], 0.45 * case["n_e"] * case["a0"] * case["fwhm_fs"] / 30.0
        inside = min(case["steps"], 1650.0 * case["fwhm_fs"] / 30.0)
        return {"bytes": b * (2.0 * n + made), "flops": 150.0 * n * inside + 90.0 * 0.5 * made * inside
                + 6.0 * (n + made) * (case["steps"] - inside)}
    lep = case["n_e"] + case["n_p"]
    rate = {"lp": 1.1e-3 * 0.5 * case.get("strength", 0.0), "cp": 0.3, "uniform": 0.014, "rotating": 0.1}.get(
        case.get("field"), 0.014)
    made = lep * case["steps"] * min(rate, 0.5)
    return {"bytes": b * (2.0 * (lep + case["n_g"]) + made),
            "flops": case["steps"] * (150.0 * lep + 90.0 * (case["n_g"] + 0.5 * made))}


# ------------------------------------------------------------------------------------- exact
# The step of Ridgers et al. (arXiv:1311.5551, Sec. 3) in 64 bits, written with torch and numpy
# alone: tables by quadrature of the integral representations of the Bessel functions, fields,
# Boris push, rates, inverse-CDF samples, recoil, pairs, and the order and the random numbers of
# the package's interface (Philox4x64-10 keyed by seed and scenario, counted by id, step, species).
def _bessel(y, nu, integral=False):
    """K_nu(y), or the integral of K_nu from y to infinity: trapezoid rule in t."""
    out = torch.zeros_like(y)
    h = 0.1
    for j in range(560):
        t = j * h
        c = math.cosh(t)
        out += torch.exp(-y * c) * ((0.5 if j == 0 else 1.0) * h * math.cosh(nu * t) / (c if integral else 1.0))
    return out


def _emissivity(eta, xi, om):
    y = 2.0 * xi / (3.0 * eta * om)
    return xi * xi * y * _bessel(y, 2.0 / 3.0) + om * y * _bessel(y, 5.0 / 3.0, True)


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return (torch.tensor(v, device="cuda") for v in (x, w))


def _panels(f, a, b, n=8):
    """Gauss-Legendre integrals of f over [a, b] (tensors), one panel each."""
    x, w = _gauss(n)
    half, mid = 0.5 * (b - a), 0.5 * (a + b)
    return (f(mid[..., None] + half[..., None] * x) * w).sum(-1) * half


_EXACT_TABLES = {}


def _exact_tables():
    if _EXACT_TABLES:
        return _EXACT_TABLES
    dev, n = "cuda", 256
    eta = torch.exp(torch.linspace(math.log(1e-4), math.log(1e2), n, device=dev, dtype=torch.float64))
    e1, e2 = eta[:, None], eta[:, None, None]

    def below(xi, power):  # integral of F xi^(power) dxi below xi, in s = xi^(1/3)
        def f(s):
            x = s ** 3
            v = 3.0 * _emissivity(e1, x, 1.0 - x)
            return v * s * s if power == 0 else v / s
        return _panels(f, torch.zeros_like(xi), xi ** (1.0 / 3.0), 16)

    def zeta(z, with_xi):  # F (1 - xi) [xi] at xi = logistic(z)
        om = 1.0 / (1.0 + torch.exp(z))
        x = 1.0 / (1.0 + torch.exp(-z))
        v = _emissivity(e2, x, om) * om
        return v * x if with_xi else v

    zhi = torch.log(90.0 * eta)
    za = math.log(1e-13)
    tiny = torch.full_like(eta, 1e-13)
    total = below(tiny, 0)
    edges = torch.arange(0, int(math.ceil((float(zhi.max()) + 6.0 - za) * 8.0)), device=dev, dtype=torch.float64) * 0.125 + za
    keep = edges[None, :] < (zhi + 6.0)[:, None]
    lo = edges[None, :].expand(n, -1)
    total = total + (_panels(lambda z: zeta(z, True), lo, lo + 0.125) * keep).sum(1)
    lx = torch.full_like(eta, math.log(1e-9))
    for _ in range(25):  # the cut-off below which photons carry 1e-9 of the energy
        x = torch.exp(lx)
        eb = below(x, 0)
        slope = x * _emissivity(eta, x, 1.0 - x) / eb
        lx = lx - ((torch.log(eb / total) - math.log(1e-9)) / slope).clamp(-3.0, 3.0)
    xmin = torch.exp(lx)
    zlo = torch.log(xmin / (1.0 - xmin))
    node = zlo[:, None] + (zhi - zlo)[:, None] * torch.arange(n, device=dev, dtype=torch.float64) / (n - 1)
    seg = _panels(lambda z: zeta(z, False), node[:, :-1], node[:, 1:])
    ends = torch.stack([zhi, zhi + 3.0], 1)
    above = _panels(lambda z: zeta(z, False), ends, ends + 3.0).sum(1)
    low = below(xmin, -1)
    h = low + above + seg.sum(1)
    zero = torch.zeros((n, 1), device=dev, dtype=torch.float64)
    P = (low[:, None] + torch.cat([zero, seg.cumsum(1)], 1)) / h[:, None]
    Q = (above[:, None] + torch.cat([seg.flip(1).cumsum(1).flip(1), zero], 1)) / h[:, None]
    chi = torch.exp(torch.linspace(math.log(1e-2), math.log(1e2), n, device=dev, dtype=torch.float64))
    lnT = torch.log(0.16 * _bessel_scaled(2.0 / (3.0 * chi)) ** 2 / chi) - 4.0 / (3.0 * chi)
    s = (0.5 * torch.arange(128, device=dev, dtype=torch.float64) / 127.0) ** (1.0 / 3.0)
    mid = 0.5 * (s[:-1] + s[1:])

    def pf(v):
        f = v ** 3
        q = f * (1.0 - f)
        return 3.0 * v * v * (2.0 + q) / q * _bessel(1.0 / (3.0 * chi[:, None, None] * q), 2.0 / 3.0)

    a, m, b = (v[None, :].expand(n, -1) for v in (s[:-1], mid, s[1:]))
    part = _panels(pf, a, m, 16) + _panels(pf, m, b, 16)
    Pf = torch.cat([zero, part.cumsum(1)], 1) / part.sum(1, keepdim=True)
    Pf[:, -1] = 1.0
    _EXACT_TABLES.update(lnh=torch.log(h), P=P, Q=Q, zlo=zlo, zhi=zhi, lnT=lnT, Pf=Pf)
    return _EXACT_TABLES


def _bessel_scaled(y):
    """exp(y) K_{1/3}(y) (y up to 67: the plain form would lose digits to underflow)."""
    out = torch.zeros_like(y)
    for j in range(400):
        t = j * 0.025
        out += torch.exp(-y * (math.cosh(t) - 1.0)) * ((0.5 if j == 0 else 1.0) * 0.025 * math.cosh(t / 3.0))
    return out


def _cell(v, lo, hi, n=256):
    s = (torch.log(v) - math.log(lo)) * ((n - 1) / (math.log(hi) - math.log(lo)))
    sc = s.clamp(min=0.0)
    i = sc.long().clamp(max=n - 2)
    return s, i, (sc - i).clamp(max=1.0)


def _lookup(table, v, lo, hi):
    _, i, w = _cell(v, lo, hi)
    return torch.exp(w * table[i + 1] + (1.0 - w) * table[i])


def _rate_T(T, chi):
    out = _lookup(T["lnT"], chi.clamp(min=1e-2), 1e-2, 1e2)
    top = torch.exp(T["lnT"][-1]) * (chi / 1e2) ** (-1.0 / 3.0)
    return torch.where(chi >= 1e-2, torch.where(chi > 1e2, top, out), torch.zeros_like(chi))


def _xi_row(T, r, U, V):
    P, Q = T["P"][r], T["Q"][r]
    n = P.shape[1]
    low = (P < U[:, None]).sum(1).sub(1).clamp(0, n - 2)
    high = (Q > V[:, None]).sum(1).sub(1).clamp(0, n - 2)
    at = lambda A, i: A.gather(1, i[:, None])[:, 0]  # noqa: E731
    p0, p1, q0, q1 = at(P, low), at(P, low + 1), at(Q, high), at(Q, high + 1)
    lower = U <= 0.5
    j = torch.where(lower, low, high)
    f = torch.where(lower, (U - p0) / (p1 - p0), (q0 - V) / (q0 - q1))
    first, last = U <= P[:, 0], V <= Q[:, -1]
    j = torch.where(first, torch.zeros_like(j), torch.where(last, torch.full_like(j, n - 2), j))
    f = torch.where(first, torch.zeros_like(f), torch.where(last, torch.ones_like(f), f))
    z = lambda k: 1.0 / (1.0 + torch.exp(-(T["zlo"][r] + k * (T["zhi"] - T["zlo"])[r] / (n - 1))))  # noqa: E731
    return z(j) + f * (z(j + 1) - z(j))


def _f_row(T, r, V):
    P = T["Pf"][r]
    n = P.shape[1]
    j = (P < V[:, None]).sum(1).sub(1).clamp(0, n - 2)
    p0, p1 = P.gather(1, j[:, None])[:, 0], P.gather(1, j[:, None] + 1)[:, 0]
    return 0.5 * (j + (V - p0) / (p1 - p0)) / (n - 1)


def _philox(ids, step, kind, purpose, seed, scen):
    """Uniforms U0..U3 of Philox4x64-10 (Salmon et al., SC'11), (m + 1/2) 2^-52."""
    def mul(a, b):
        lo32 = np.uint64(0xFFFFFFFF)
        s = np.uint64(32)
        al, ah, bl, bh = a & lo32, a >> s, b & lo32, b >> s
        m1, m2 = ah * bl, al * bh
        mid = ((al * bl) >> s) + (m1 & lo32) + (m2 & lo32)
        return a * b, ah * bh + (m1 >> s) + (m2 >> s) + (mid >> s)

    c = [np.asarray(ids, dtype=np.uint64)] + [np.full(len(ids), v, dtype=np.uint64) for v in (step, kind, purpose)]
    k0, k1 = seed, scen
    for _ in range(10):
        lo0, hi0 = mul(c[0], np.uint64(0xD2E7470EE14C6C93))
        lo1, hi1 = mul(c[2], np.uint64(0xCA5A826395121157))
        c = [hi1 ^ c[1] ^ np.uint64(k0), lo1, hi0 ^ c[3] ^ np.uint64(k1), lo0]
        k0, k1 = (k0 + 0x9E3779B97F4A7C15) % 2 ** 64, (k1 + 0xBB67AE8584CAA73B) % 2 ** 64
    return [torch.tensor(((w >> np.uint64(12)).astype(np.float64) + 0.5) * 2.0 ** -52, device="cuda") for w in c]


def _gather(grid, shape, org, spc, x):
    """Yee-staggered grid fields at the particles, linear (1) or quadratic (2) weights."""
    n = (grid.shape[3], grid.shape[2], grid.shape[1])
    g = grid.double()

    def weights(a, half):
        s = (x[a] - org[a]) / spc[a] - (0.5 if half else 0.0)
        if shape == 1:
            i = torch.floor(s)
            return i.long(), [1.0 - (s - i), s - i]
        i = torch.round(s)
        d = s - i
        return i.long() - 1, [0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2]

    out = []
    for c in range(6):
        half = [(a == c) if c < 3 else (a != c - 3) for a in range(3)]
        ws = [weights(a, half[a]) for a in range(3)]
        v = torch.zeros_like(x[0])
        for dz, wz in enumerate(ws[2][1]):
            for dy, wy in enumerate(ws[1][1]):
                for dx, wx in enumerate(ws[0][1]):
                    i = [ws[0][0] + dx, ws[1][0] + dy, ws[2][0] + dz]
                    ok = (i[0] >= 0) & (i[0] < n[0]) & (i[1] >= 0) & (i[1] < n[1]) & (i[2] >= 0) & (i[2] < n[2])
                    j = [i[a].clamp(0, n[a] - 1) for a in range(3)]
                    v = v + torch.where(ok, wx * wy * wz * g[c, j[2], j[1], j[0]], torch.zeros_like(v))
        out.append(v)
    return out[:3], out[3:]


def _fields(fld, t, x0, v, x):
    zero = torch.zeros_like(x[0])
    if fld["kind"] == qed.FIELD_UNIFORM:
        return [zero] * 3, [zero + b for b in fld["B"]]
    if fld["kind"] == qed.FIELD_ROTATING_E:
        ph = fld["omega"] * t
        return [zero + fld["E0"] * math.cos(ph), zero + fld["E0"] * math.sin(ph), zero], [zero] * 3
    if fld["kind"] == qed.FIELD_GRID:
        return _gather(fld["grid"], fld["shape"], fld["origin"], fld["spacing"], x)
    phi = fld["omega"] * (t - (x0 + v * t) - x[0]) - fld.get("phi_start", 0.0)
    env, L = zero + 1.0, fld.get("phi_len", 0.0)
    if L > 0.0:
        env = torch.where((phi > 0.0) & (phi < L), torch.sin(math.pi * phi / L) ** 2, zero)
    ec, es = fld["E0"] * env * torch.cos(phi), fld["E0"] * env * torch.sin(phi)
    if fld["kind"] == qed.FIELD_PLANE_LP:
        return [zero, ec, zero], [zero, zero, ec]
    return [zero, ec, es], [zero, -es, ec]


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _invariant(u, en, E, B):
    """sqrt((en E + u x B)^2 - (u.E)^2); in a plane wave along x the cancellation-free product."""
    f = [en * E[c] + v for c, v in enumerate(_cross(u, B))]
    return torch.sqrt((_dot(f, f) - _dot(u, E) ** 2).clamp(min=0.0))


def _wave_invariant(u, en, E, massive):
    d = torch.where(u[0] > 0.0, (u[1] ** 2 + u[2] ** 2 + massive) / (en + u[0]), en - u[0])
    return d * torch.sqrt(_dot(E, E))


def _simulate(sets, drained, fld, dt, x0, v, first, steps, seed, scen, emit, pairs, drain, recoil):
    """sets: per species (e-, e+, photons) [x(3), u(3), tau, id] in FP64; steps it in place."""
    T = _exact_tables()
    wave = fld["kind"] in (qed.FIELD_PLANE_LP, qed.FIELD_PLANE_CP)
    nid = [s[7].numel() for s in sets] + [0]
    led = []
    for step in range(first, first + steps):
        t = step * dt
        born = {0: [], 1: [], 2: []}
        n_emit = e_emit = n_pair = e_pair = 0.0
        for k in (0, 1):
            s = sets[k]
            if not s[0].numel():
                continue
            q = -1.0 if k == 0 else 1.0
            x, u = s[:3], s[3:6]
            E, B = _fields(fld, t, x0, v, x)
            m = [u[c] + 0.5 * q * dt * E[c] for c in range(3)]
            tb = [0.5 * q * dt / torch.sqrt(1.0 + _dot(m, m)) * B[c] for c in range(3)]
            sb = [2.0 / (1.0 + _dot(tb, tb)) * tb[c] for c in range(3)]
            mp = [m[c] + w for c, w in enumerate(_cross(m, tb))]
            u = [m[c] + w + 0.5 * q * dt * E[c] for c, w in enumerate(_cross(mp, sb))]
            gam = torch.sqrt(1.0 + _dot(u, u))
            x = [x[c] + dt * (u[c] / gam - (v if c == 0 else 0.0)) for c in range(3)]
            eta = _wave_invariant(u, gam, E, 1.0) if wave else _invariant(u, gam, E, B)
            lam = math.sqrt(3.0) * ALPHA / (2.0 * math.pi) * eta / gam * _lookup(T["lnh"], eta.clamp(min=1e-300), 1e-4, 1e2)
            s[6] = s[6] - torch.where(eta > 0.0, lam * dt, torch.zeros_like(lam))
            if emit:
                ev = torch.nonzero(s[6] <= 0.0)[:, 0]
                U = _philox(s[7][ev].cpu().numpy(), step, k, 0, seed, scen)
                ge, ue = gam[ev], [c[ev] for c in u]
                sv, i, w = _cell(eta[ev], 1e-4, 1e2)
                ok = U[0] >= (1.0 - w) * T["P"][i, 0] + w * T["P"][i + 1, 0]
                xi = (1.0 - w) * _xi_row(T, i, U[0], 1.0 - U[0]) + w * _xi_row(T, i + 1, U[0], 1.0 - U[0])
                xi = torch.where(sv < 0.0, xi * eta[ev] / 1e-4, xi).clamp(max=1.0)
                eps = xi * ge
                um = torch.sqrt(_dot(ue, ue))
                uf = torch.sqrt(((ge - eps) ** 2 - 1.0).clamp(min=0.0)) if recoil else (um - eps).clamp(min=0.0)
                for c in range(3):
                    u[c][ev] = torch.where(ok, uf * ue[c] / um, ue[c])
                s[6][ev] = -torch.log(U[1])
                born[2].append([c[ev][ok] for c in x] + [(eps * c / um)[ok] for c in ue] + [-torch.log(U[2][ok])])
                n_emit += float(ok.sum())
                e_emit += float(eps[ok].sum())
            s[:6] = x + u
        s = sets[2]
        if s[0].numel():
            x, kk = s[:3], s[3:6]
            live = torch.isfinite(s[6])
            E, B = _fields(fld, t, x0, v, x)
            eps = torch.sqrt(_dot(kk, kk))
            chi = 0.5 * (_wave_invariant(kk, eps, E, 0.0) if wave else _invariant(kk, eps, E, B))
            s[6] = s[6] - ALPHA * chi / eps * _rate_T(T, chi) * dt
            for c in range(3):
                s[c] = torch.where(live, x[c] + dt * (kk[c] / eps - (v if c == 0 else 0.0)), x[c])
            if pairs:
                ev = torch.nonzero(s[6] <= 0.0)[:, 0]
                if ev.numel():
                    U = _philox(s[7][ev].cpu().numpy(), step, 2, 0, seed, scen)
                    _, i, w = _cell(chi[ev], 1e-2, 1e2)
                    lower = U[0] < 0.5
                    V = torch.where(lower, 2.0 * U[0], 2.0 * (1.0 - U[0]))
                    f = (1.0 - w) * _f_row(T, i, V) + w * _f_row(T, i + 1, V)
                    f = torch.where(lower, f, 1.0 - f)
                    ee, xe, ke = eps[ev], [s[c][ev] for c in range(3)], [c[ev] for c in kk]
                    share = [1.0 - f, f]
                    if recoil:
                        kin = (ee - 2.0).clamp(min=0.0)
                        share = [torch.where(ee >= 2.0, torch.sqrt((1.0 + p * kin) ** 2 - 1.0) / ee, p) for p in share]
                    for d in (0, 1):
                        born[d].append(xe + [share[d] * c for c in ke] + [-torch.log(U[1 + d])])
                    s[6][ev] = math.inf
                    n_pair += ev.numel()
                    e_pair += float(ee.sum())
        for d in (0, 1, 2):
            new = [torch.cat(c) for c in zip(*born[d])] if born[d] else None
            dst = drained if d == 2 and drain else sets[d]
            slot = 3 if d == 2 and drain else d
            if new is not None and new[0].numel():
                m = new[0].numel()
                ids = torch.arange(nid[slot], nid[slot] + m, device="cuda", dtype=torch.int64)
                dst[:] = [torch.cat([a, b]) for a, b in zip(dst, new + [ids])]
                nid[slot] += m
        led = [n_emit, e_emit, float(n_pair), e_pair]
    held = [torch.isfinite(s[6]) for s in sets]
    energy = [float(torch.sqrt((1.0 if k < 2 else 0.0) + _dot(s[3:6], s[3:6]))[h].sum())
              for k, (s, h) in enumerate(zip(sets, held))]
    return np.array([float(h.sum()) for h in held] + energy + led)


def _as_outputs(s, n, cap, mixed, name):
    """As _held: the particles that went in and the room for new ones.  In the mixed path a new
    particle's place depends on every earlier event, so new ones have no value here; nor has the
    low part of an optical depth (the rounding that the leading float leaves)."""
    cols = dict(zip((*_COLS, "tau"), s[:7]))
    out = {}
    if n:
        out[name] = {k: t[:n] for k, t in cols.items()}
    if n < cap:
        out["new_" + name] = {k: None if mixed else torch.nn.functional.pad(t[n:], (0, cap - t.numel()))
                              for k, t in cols.items()}
    return out


def _start_set(cols):
    n = cols[0].numel()
    return [c.double() for c in cols] + [torch.arange(n, device="cuda", dtype=torch.int64)]


def _exact_merge(case, seed):
    cols, span = _merge_inputs(case, seed)
    a = np.stack([c.double().cpu().numpy() for c in cols])
    x, k = a[:3], a[3:6]
    cell = 2.0 * span / case["cells"]
    ci = np.floor((x + span) / cell)
    inside = np.all((ci >= 0) & (ci < case["cells"]), axis=0)
    ax = np.argmax(np.abs(k), axis=0)
    big = np.take_along_axis(k, ax[None], 0)[0]
    bins = np.clip(np.floor((k / np.abs(big) + 1.0) * 0.5 * case["n_face"]), 0, case["n_face"] - 1)
    others = np.array([[1, 2], [0, 2], [0, 1]])[ax].T
    face = np.take_along_axis(bins, others, 0)
    en = np.sqrt(k[0] * k[0] + k[1] * k[1] + k[2] * k[2])
    mant, ex = np.frexp(en)
    sub = np.minimum(np.floor((mant - 0.5) * 2.0 * case["n_sub"]), case["n_sub"] - 1)
    key = (ci[2] * case["cells"] + ci[1]) * case["cells"] + ci[0]
    for part, size in ((2 * ax + (big < 0), 6), (face[0], case["n_face"]), (face[1], case["n_face"]), (ex + 1100, 2200),
                       (sub, case["n_sub"])):
        key = key * size + part
    key = np.where(inside, key, -1.0).astype(np.int64)
    order = np.argsort(key, kind="stable")
    order = order[np.searchsorted(key[order], 0):]
    starts = np.flatnonzero(np.diff(key[order], prepend=-2))
    sizes = np.diff(np.append(starts, len(order)))
    total = lambda v: np.add.reduceat(v[order], starts)  # noqa: E731
    big_enough = sizes >= case["min_group"]
    W, E = sizes.astype(np.float64), total(en)
    mv, mx = np.stack([total(c) for c in k]) / W, np.stack([total(c) for c in x]) / W
    et = E / W
    dl = np.sqrt(np.maximum(et * et - (mv * mv).sum(0), 0.0))
    small = np.argmin(np.abs(mv), axis=0)
    unit = np.zeros_like(mv)
    np.put_along_axis(unit, small[None], 1.0, 0)
    dv = np.cross(mv, unit, axis=0)
    norm = np.sqrt((dv * dv).sum(0))
    dv = np.where(norm > 0, dv * dl / np.where(norm > 0, norm, 1.0), unit * dl)
    gone = np.zeros(a.shape[1], dtype=bool)
    member = np.repeat(big_enough, sizes) & (np.arange(len(order)) - np.repeat(starts, sizes) >= 2)
    gone[order[member]] = True
    for j, sign in ((0, 1.0), (1, -1.0)):
        i = order[starts[big_enough] + j]
        a[:3, i], a[3:6, i] = mx[:, big_enough], (mv + sign * dv)[:, big_enough]
    left = a[:, ~gone]
    left = np.pad(left, ((0, 0), (0, a.shape[1] - left.shape[1])))
    return {"groups": int(big_enough.sum()), "photons": dict(zip((*_COLS, "tau"), left))}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("job", "batch"):
        return None  # thousands of steps (hundreds, of many scenarios): minutes in plain torch
    if kind == "merge":
        return _exact_merge(case, seed)
    mixed = case["prec"] == "mixed"
    opt = dict(emit=True, pairs=case.get("pairs", True), drain=case.get("drain", False), recoil=case.get("recoil", False))
    sets = [_start_set(c) for c in _inputs(case, seed)]
    drained = _start_set([c[:0] for c in _inputs(case, seed)[0]])
    if kind == "steps":
        fld, dt, first, x0, v = _setting(case)
    elif kind == "pic":
        grid, org, spc = _grid_field(case, seed)
        fld = dict(kind=qed.FIELD_GRID, grid=grid, shape=case["shape"], origin=org, spacing=spc)
        dt, first, x0, v = 2.0 * math.pi * 1e6 / 1000.0, 0, 0.0, 0.0
    else:
        fld, first, x0, v = dict(kind=qed.FIELD_UNIFORM, B=(0.0, 0.0, case["strength"])), 0, 0.0, 0.0
        dt = 2.0 * math.pi * case["gamma"] / case["strength"] / 1000.0
        opt.update(pairs=False, drain=True)
    led = _simulate(sets, drained, fld, dt, x0, v, first, case["steps"], int(seed), 0, **opt)
    e_cap, p_cap, g_cap = _step_caps(case) if kind != "noalloc" else (case["n"], 0, case["n"] * case["steps"] + 64)
    n_in = (case.get("n_e", case.get("n")), case.get("n_p", 0), case.get("n_g", 0))
    if opt["drain"]:
        e = _as_outputs(sets[0], n_in[0], e_cap, mixed, "electrons")
        if kind == "noalloc":
            return {**e, "photons": _as_outputs(drained, 0, g_cap, mixed, "p")["new_p"]}
        return {**e, **_as_outputs(drained, 0, g_cap, mixed, "drained"), "ledger": led}
    out = {"ledger": led}
    for s, n, cap, name in zip(sets, n_in, (e_cap, p_cap, g_cap), _NAMES):
        out.update(_as_outputs(s, n, cap, mixed, name))
    return out
