"""The merge of a step's children into (parent species, parent index) order, at the edges of the
groups that its ranks are summed over (32 particles per mask word, 1024 per fine group, 32768 per
coarse group): every new photon sits at its parent's position, in parent order, with the next
ids.  Exact comparisons: a photon is created at its parent's position."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1311_5551_gb300 import build as qbuild  # noqa: E402
from paper_1311_5551_gb300 import qed  # noqa: E402


@pytest.fixture(scope="module")
def tables():
    qbuild.build()
    return qed.Tables()


def species(prec, cap):
    return [qed.Species(qed.ELECTRON, prec, cap, cap), qed.Species(qed.POSITRON, prec, cap, cap),
            qed.Species(qed.PHOTON, prec, 8 * cap, 2 * cap)]


def load(sp, ns, seed):
    """ns[k] leptons of kind k on a line, a tenth of them about to emit."""
    rng = np.random.default_rng(seed)
    for k, n in enumerate(ns):
        x = np.zeros((n, 3))
        x[:, 0] = 4096.0 * (np.arange(n) + k * 200000)
        u = np.tile([[1000.0, 0.0, 0.0]], (n, 1))
        sp[k].upload(x, u, tau=np.where(rng.random(n) < 0.1, 1e-9, 50.0))
    sp[2].upload(np.zeros((0, 3)), np.zeros((0, 3)))


def step_and_check(tables, sp, params, step, run):
    before = sp[2].count()
    tau0 = [s.download()["tau"] for s in sp[:2]]
    run(step)
    qed.check(sp)
    g = sp[2].download()
    parents = []
    for s, t in zip(sp[:2], tau0):
        d = s.download()
        # the optical depth only grows when it is drawn afresh after an event; an event below the
        # energy cut makes no photon and leaves the momentum's size as it was
        emitted = (d["tau"] > t) | (t < 1e-8)
        size = np.linalg.norm(d["u"].astype(np.float64), axis=1)
        parents.append(d["x"][emitted & (size < 999.9)])
    want = np.concatenate(parents)
    made = np.flatnonzero(np.arange(len(g["id"])) >= before)
    sure = np.isin(g["x"][made][:, 0], want[:, 0])
    assert len(want) and np.array_equal(g["x"][made][sure], want)  # in order, none missing
    assert np.array_equal(g["id"][made], np.arange(before, before + len(made)))
    # every photon has a parent; the few softest ones left it almost at its old momentum
    every = np.concatenate([s.download()["x"] for s in sp[:2]])
    where = np.searchsorted(every[:, 0], g["x"][made][:, 0])
    assert np.all(np.diff(where) > 0) and np.array_equal(every[where], g["x"][made])


@pytest.mark.parametrize("prec", [qed.MIXED, qed.FP64])
@pytest.mark.parametrize("ns", [(33, 31), (1023, 1025), (1024, 0), (32767, 40), (32769, 32800), (70001, 1)])
def test_children_in_parent_order(tables, prec, ns):
    sp = species(prec, sum(ns) + 64)
    p = qed.StepParams(dt=10.0, seed=3, field=qed.Field(B=(0.0, 0.0, 1e-3)), make_pairs=False)
    load(sp, ns, 5)
    step_and_check(tables, sp, p, 0, lambda k: qed.run(tables, sp, p, k))


def test_counts_are_cleared_between_populations(tables):
    # large, small, then large again: the event counts of earlier steps leave nothing behind, on
    # the single path and in a batch
    prec = qed.MIXED
    sp = species(prec, 70000)
    p = qed.StepParams(dt=10.0, seed=4, field=qed.Field(B=(0.0, 0.0, 1e-3)), make_pairs=False)
    batch = qed.Batch(tables, prec, 2)

    def in_batch(step):
        batch.attach(1, sp, p, step, 1)
        batch.run(1)

    for seed, ns in enumerate([(60000, 1500), (40, 10), (50, 1), (65000, 2000), (33000, 33000)]):
        load(sp, ns, seed)
        step_and_check(tables, sp, p, seed, (lambda k: qed.run(tables, sp, p, k)) if seed % 3 else in_batch)


@pytest.mark.parametrize("parent", [qed.ELECTRON, qed.PHOTON])
def test_order_beyond_1024_coarse_groups(tables, parent):
    # more than 1024 x 32768 parents: the merge's prefixes stand for two coarse groups each.  Every 37th
    # parent has an event; a child starts at its parent's position, which tells whose it is
    n = 34_000_037
    i = torch.arange(n, device="cuda", dtype=torch.int64)
    x = torch.stack([(i % 4099).float() * 3.0, (i % 509).float(), (i // 37).float()], dim=1)
    u = torch.zeros((n, 3), device="cuda")
    u[:, 0] = 1e3 if parent == qed.ELECTRON else 1e5
    has = i % 37 == 5
    tau = torch.where(has, 1e-12, 1e3).double()
    want = int(has.sum())
    cap = {k: n if k == parent else want + 10 for k in (qed.ELECTRON, qed.POSITRON, qed.PHOTON)}
    sp = [qed.Species(k, qed.MIXED, cap[k], want + 10) for k in (qed.ELECTRON, qed.POSITRON, qed.PHOTON)]
    src = sp[0 if parent == qed.ELECTRON else 2]
    src.upload(x, u, tau=tau)
    qed.run(tables, sp, qed.StepParams(dt=10.0, seed=4, field=qed.Field(B=(0.0, 0.0, 1e-3))), 0, 1)
    qed.check(sp)
    led = qed.read_ledger(sp)
    at = src.download()["x"][5::37]  # the parents after the push, in order
    if parent == qed.ELECTRON:
        kids = [sp[2].download()]
        assert led["emitted_n"] + led["dropped_n"] == want and len(kids[0]["id"]) == led["emitted_n"] > 0.9 * want
    else:
        kids = [sp[0].download(), sp[1].download()]
        assert led["pairs_n"] == want and all(len(c["id"]) == want for c in kids)
    for c in kids:
        who = np.round(c["x"][:, 2]).astype(np.int64)
        assert np.all(np.diff(who) > 0)
        assert np.array_equal(c["x"], at[who])
        assert np.array_equal(c["id"], np.arange(len(who), dtype=np.uint32))
