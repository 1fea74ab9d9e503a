"""Runs that take their photons several steps at a time (windows) against the same steps one call
at a time, which never form a window: the particles, ids, weights and work counters are the same
bit for bit, in every kind of field, around the sizes at which windows begin (1024 photons) and
end (16 steps), with photons that convert, were converted, or start without optical depth."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1311_5551_gb300 import build as qbuild  # noqa: E402
from paper_1311_5551_gb300 import qed  # noqa: E402

DT = 2.0e4


@pytest.fixture(scope="module")
def tables():
    qbuild.build()
    return qed.Tables()


def field(kind):
    if kind == "uniform":
        return qed.Field(E=(2e-4, 0.0, 1e-4), B=(0.0, 3e-4, 1e-3))
    if kind == "rotating":
        return qed.Field(kind=qed.FIELD_ROTATING_E, E0=1e-3, omega=3e-6)
    if kind == "lp":  # a pulse a few steps long: photons enter and leave it within the run
        return qed.Field(kind=qed.FIELD_PLANE_LP, E0=1e-3, omega=2e-5, phi_start=-2.0, phi_len=12.0)
    if kind == "cp":
        return qed.Field(kind=qed.FIELD_PLANE_CP, E0=1e-3, omega=2e-6)
    g = torch.tensor(np.random.default_rng(1).normal(size=(6, 7, 8, 9)) * 1e-3, dtype=torch.float32, device="cuda")
    return qed.Field(kind=qed.FIELD_GRID, grid=g, shape=2 if kind == "tsc" else 1, origin=(-4e5,) * 3, spacing=(1e5,) * 3)


def population(seed, n_e, n_g, weights):
    rng = np.random.default_rng(seed)
    sp = [qed.Species(qed.ELECTRON, qed.MIXED, 4 * (n_e + n_g) + 64, n_e + n_g),
          qed.Species(qed.POSITRON, qed.MIXED, 4 * (n_e + n_g) + 64, n_e + n_g),
          qed.Species(qed.PHOTON, qed.MIXED, 120 * (n_e + n_g) + 64, 4 * (n_e + n_g))]

    def vectors(n, size):
        d = rng.normal(size=(n, 3))
        return d / np.linalg.norm(d, axis=1, keepdims=True) * size[:, None]

    sp[0].upload(rng.normal(size=(n_e, 3)) * 2e5, vectors(n_e, rng.uniform(100, 3000, n_e)))
    sp[0].init_tau(seed)
    # energies from far below the tables to far above: no rate, a small one, frequent conversions
    tau = rng.exponential(size=n_g)
    tau[::7] *= 1e-2
    tau[3::211] = 0.0       # used up before the first step
    tau[5::101] = np.inf    # converted earlier
    sp[2].upload(rng.normal(size=(n_g, 3)) * 2e5, vectors(n_g, 10.0 ** rng.uniform(-1, 6, n_g)), tau=tau)
    if weights:
        sp[2].set_weights(rng.uniform(0.5, 2.0, n_g))
    return sp


@pytest.mark.parametrize("kind", ["uniform", "rotating", "lp", "cp", "cic", "tsc"])
@pytest.mark.parametrize("n_g,steps", [(1023, 6), (1024, 2), (1025, 3), (3071, 17), (2048, 18), (5000, 35)])
def test_windows_match_single_steps(tables, kind, n_g, steps):
    p = qed.StepParams(dt=DT, t0=-10 * DT, seed=11, field=field(kind), window_x0=100.0, window_v=-0.5)
    first = 5
    runs = []
    for window in (False, True):
        sp = population(3, 500, n_g, weights=steps == 18)
        if window:
            qed.run(tables, sp, p, first, steps)
        else:
            for k in range(steps):
                qed.run(tables, sp, p, first + k, 1)
        qed.check(sp)
        runs.append((sp, qed.work_read(sp[0])))
    (ref, wr), (got, wg) = runs
    for a, b in zip(ref, got):
        assert np.array_equal(a.save(), b.save())
    assert wr == wg
    # the last step's sums run over the same particles in the same order; only the electrons that a
    # window's conversions made sit in the ledger as they do on the single steps
    assert qed.read_ledger(ref) == qed.read_ledger(got)
    assert ref[1].count() > 0  # photons converted


def test_windows_respect_the_switches(tables):
    # no pair creation, and photons drained: the photons already held still move and lose nothing
    for opt in (dict(make_pairs=False), dict(drain_photons=True), dict(emit_photons=False, recoil_energy=True)):
        p = qed.StepParams(dt=DT, seed=5, field=field("rotating"), **opt)
        out = []
        for window in (False, True):
            sp = population(4, 300, 2100, weights=False) + [qed.Species(qed.PHOTON, qed.MIXED, 50000, 1)]
            for k in range(0, 20, 20 if window else 1):
                qed.run(tables, sp, p, k, 20 if window else 1)
            qed.check(sp)
            out.append([s.save() for s in sp])
        assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("graph_steps", [0, 8, 32])
def test_batch_windows_match_single_runs(tables, graph_steps):
    # slots of every field, with different steps left, advanced by calls that end inside and at the
    # end of a graph: each slot's particles and ledger are those of its own run
    kinds = ["uniform", "rotating", "lp", "cp", "lp", "rotating"]
    sizes = [(1023, 40), (5000, 37), (3071, 17), (2048, 2), (1100, 1), (20000, 40)]
    first = 5

    def params(k):
        return qed.StepParams(dt=DT, t0=-10 * DT, seed=11, scenario=k, field=field(kinds[k]), window_x0=100.0,
                              window_v=-0.5)

    refs = []
    for k, (n_g, steps) in enumerate(sizes):
        sp = population(20 + k, 400, n_g, weights=k == 1)
        qed.run(tables, sp, params(k), first, steps)
        refs.append((sp, qed.work_read(sp[0])))
    batch = qed.Batch(tables, qed.MIXED, len(sizes) + 1)
    batch.config(0, graph_steps)
    mix = [population(20 + k, 400, n_g, weights=k == 1) for k, (n_g, _) in enumerate(sizes)]
    for k, sp in enumerate(mix):
        batch.attach(k, sp, params(k), first, sizes[k][1])
    for n in (8, 1, 2, 16, 3, 32):
        batch.run(n)
    assert np.all(batch.remaining() == 0)
    for k, ((ref, wr), sp) in enumerate(zip(refs, mix)):
        qed.check(sp)
        for a, b in zip(ref, sp):
            assert np.array_equal(a.save(), b.save()), f"slot {k}"
        assert qed.read_ledger(ref) == qed.read_ledger(sp)
        assert wr == qed.work_read(sp[0])
