"""The inverse-CDF samples through the device tables' guides against the definition (the largest node
below the draw, found here by a plain binary search over the row): few and many nodes, plateaus,
draws on the guides' edges, and rows that are not monotone, where the whole row is searched."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1311_5551_gb300 import build as qbuild  # noqa: E402
from paper_1311_5551_gb300 import qed  # noqa: E402

N_ETA, N_CHI = 5, 4


def make(n_xi, n_f, rng, broken):
    def cdf(n):
        # steps over many decades, some of them zero (plateaus)
        s = 10.0 ** rng.uniform(-6, 0, n) * (rng.random(n) < 0.8)
        s[0] = 10.0 ** rng.uniform(-7, -3)
        c = np.cumsum(s)
        return c / c[-1]

    P = np.stack([cdf(n_xi) * 0.999 for _ in range(N_ETA)])
    Q = 1.0 - P
    F = np.stack([(cdf(n_f) - 0.0) for _ in range(N_CHI)])
    F[:, 0], F[:, -1] = 0.0, 1.0
    if broken and n_xi > 4:
        P[1, n_xi // 2] = 0.1 * P[1, n_xi // 2 - 1]
        Q[2, n_xi // 3] = 0.1 * Q[2, n_xi // 3 + 1]
        F[1, n_f // 2] = 0.0
    spec = qed.TableSpec(n_eta=N_ETA, eta_min=1e-2, eta_max=1e2, n_xi=n_xi, n_chi=N_CHI, chi_min=1e-2, chi_max=1e2,
                         n_f=n_f)
    arrays = dict(ln_h=np.linspace(1, 0, N_ETA), g=np.ones(N_ETA), zeta_lo=np.linspace(-20, -15, N_ETA),
                  zeta_hi=np.linspace(1, 6, N_ETA), P=P, Q=Q, ln_T=np.linspace(-9, -1, N_CHI), Pf=F)
    return spec, arrays


def cell(v, lo, hi, n):
    s = (np.log(v) - np.log(lo)) * ((n - 1) / (np.log(hi) - np.log(lo)))
    i = min(int(max(s, 0.0)), n - 2)
    return i, min(max(s, 0.0) - i, 1.0)


def search(row, below):
    lo, hi = 0, len(row) - 1
    while hi - lo > 1:
        mid = (lo + hi) >> 1
        if below(row[mid]):
            lo = mid
        else:
            hi = mid
    return lo


def xi_ref(a, spec, eta, U):
    def node(r, j):
        return 1.0 / (1.0 + np.exp(-(a["zeta_lo"][r] + j * (a["zeta_hi"][r] - a["zeta_lo"][r]) / (spec.n_xi - 1))))

    def row(r):
        P, Q, V = a["P"][r], a["Q"][r], 1.0 - U
        if U <= P[0]:
            return node(r, 0)
        if V <= Q[-1]:
            return node(r, spec.n_xi - 1)
        if U <= 0.5:
            j = search(P, lambda t: t < U)
            f = (U - P[j]) / (P[j + 1] - P[j])
        else:
            j = search(Q, lambda t: t > V)
            f = (Q[j] - V) / (Q[j] - Q[j + 1])
        return node(r, j) + f * (node(r, j + 1) - node(r, j))

    i, w = cell(eta, spec.eta_min, spec.eta_max, spec.n_eta)
    if U < (1 - w) * a["P"][i][0] + w * a["P"][i + 1][0]:
        return None
    return min((1 - w) * row(i) + (w * row(i + 1) if w > 0 else 0.0), 1.0)


def f_ref(a, spec, chi, U):
    i, w = cell(chi, spec.chi_min, spec.chi_max, spec.n_chi)
    V = 2 * U if U < 0.5 else 2 * (1 - U)

    def row(r):
        P = a["Pf"][r]
        j = search(P, lambda t: t < V)
        f = (V - P[j]) / (P[j + 1] - P[j])
        n = spec.n_f - 1
        return 0.5 * j / n + f * (0.5 * (j + 1) / n - 0.5 * j / n)

    fh = (1 - w) * row(i) + (w * row(i + 1) if w > 0 else 0.0)
    return fh if U < 0.5 else 1 - fh


@pytest.mark.parametrize("broken", [False, True])
@pytest.mark.parametrize("n_xi,n_f", [(2, 2), (3, 3), (5, 4), (64, 33), (256, 128), (1000, 700)])
def test_samples_through_guides(n_xi, n_f, broken):
    qbuild.build()
    rng = np.random.default_rng(n_xi + 7 * n_f)
    spec, arrays = make(n_xi, n_f, rng, broken)
    tables = qed.Tables(spec, arrays)
    edges = np.arange(1, 512) / 512.0
    U = np.concatenate([rng.random(1500), edges, edges + 1e-15, 10.0 ** rng.uniform(-9, -3, 300),
                        1 - 10.0 ** rng.uniform(-9, -3, 300), [0.5, np.nextafter(0.5, 1)]])
    eta = 10.0 ** rng.uniform(-2, 2, len(U))
    got, ok = qed.sample(tables, qed.FP64, 0, eta, U)
    ref = [xi_ref(arrays, spec, e, u) for e, u in zip(eta, U)]
    assert np.array_equal(ok, [r is not None for r in ref])
    fine = [k for k, r in enumerate(ref) if r is not None and np.isfinite(r)]
    np.testing.assert_allclose(got[fine], [ref[k] for k in fine], rtol=1e-12)
    got, _ = qed.sample(tables, qed.FP64, 1, eta, U)
    ref = np.array([f_ref(arrays, spec, e, u) for e, u in zip(eta, U)])
    fine = np.isfinite(ref)
    np.testing.assert_allclose(got[fine], ref[fine], rtol=1e-12)


@pytest.mark.parametrize("prec", [qed.FP64, qed.MIXED])
def test_draws_outside_the_unit_interval(prec):
    # the diagnostic takes any number as the draw: outside [0, 1] it extrapolates from the row's first
    # or last bracket, as the plain search does, and a NaN gives a NaN
    qbuild.build()
    spec, arrays = make(64, 33, np.random.default_rng(5), False)
    tables = qed.Tables(spec, arrays)
    U = np.repeat([-1e30, -1e6, -0.5, -1.0 / 512, -1e-9, 0.0, 1.0, 1 + 1e-6, 1.5, 3.0, 1e6, 1e30, np.inf, -np.inf, np.nan], 40)
    par = 10.0 ** np.random.default_rng(6).uniform(-2, 2, len(U))
    got, ok = qed.sample(tables, prec, 0, par, U)
    for e, u, g, k in zip(par, U, got, ok):
        r = xi_ref(arrays, spec, e, u)
        assert k == (r is not None)
        if r is not None:
            np.testing.assert_allclose(g, r, rtol=1e-12 if prec == qed.FP64 else 1e-4)
    if prec == qed.FP64:
        got, _ = qed.sample(tables, prec, 1, par, U)
        with np.errstate(all="ignore"):
            ref = np.array([f_ref(arrays, spec, e, u) for e, u in zip(par, U)])
        np.testing.assert_allclose(got, ref, rtol=1e-12)
