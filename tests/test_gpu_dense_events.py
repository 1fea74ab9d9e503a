"""Steps in which nearly every particle has its event: more than a block can take at once are
waiting when its tiles run out.  An optical depth is either so small that the first step uses it
up or so large that no step does, so the number of events is known exactly."""
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


# two and more tiles per block of the largest grid, a ragged last one, and less than one tile each
@pytest.mark.parametrize("n", [40, 100_000, 400_003])
@pytest.mark.parametrize("share", [0.97, 1.0])
@pytest.mark.parametrize("precision", [qed.MIXED, qed.FP64])
def test_no_event_is_left(tables, precision, share, n):
    rng = np.random.default_rng(n)
    sp = [qed.Species(qed.ELECTRON, precision, 2 * n, n), qed.Species(qed.POSITRON, precision, n, n),
          qed.Species(qed.PHOTON, precision, 2 * n, n)]
    x, u = rng.normal(size=(n, 3)), np.tile([3000.0, 0.0, 0.0], (n, 1))
    due = rng.random((2, n)) < share
    for s, kind in zip((sp[0], sp[2]), due):
        s.upload(x, u, tau=np.where(kind, 1e-9, 1e3))
    p = qed.StepParams(dt=2e4, seed=5, field=qed.Field(B=(0.0, 0.0, 1e-3)))
    qed.run(tables, sp, p, 0, 1)
    qed.check(sp)
    led = qed.read_ledger(sp)
    assert led["emitted_n"] + led["dropped_n"] == due[0].sum()
    assert led["pairs_n"] == due[1].sum()
    e, g = sp[0].download(), sp[2].download()
    assert len(e["id"]) == n + due[1].sum() and sp[1].count() == due[1].sum()
    assert np.isfinite(g["tau"]).sum() == n - due[1].sum() + led["emitted_n"]
    assert (e["tau"] > 0).all() and (g["tau"] > 0).all()


# FP64 steps take up to 8 events per warp four lanes to an event, more of them one lane each: the events
# of a few particles are the same, bit for bit, whether the others of their tile have one or not
@pytest.mark.parametrize("recoil_energy", [False, True])
@pytest.mark.parametrize("few", [1, 2, 7, 8, 9, 31, 32, 33])
def test_few_events_as_many(tables, few, recoil_energy):
    n = 128
    rng = np.random.default_rng(few)
    x = rng.normal(size=(n, 3)) * 1e5
    d = rng.normal(size=(2, n, 3))
    u = d / np.linalg.norm(d, axis=2, keepdims=True) * rng.uniform(1500.0, 30000.0, (2, n, 1))
    out = []
    for due in (few, n):
        sp = [qed.Species(qed.ELECTRON, qed.FP64, 2 * n, n), qed.Species(qed.POSITRON, qed.FP64, n, n),
              qed.Species(qed.PHOTON, qed.FP64, 2 * n, n)]
        for s, k in ((sp[0], u[0]), (sp[2], u[1])):
            s.upload(x, k, tau=np.where(np.arange(n) < due, 1e-9, 1e3))
        p = qed.StepParams(dt=2e4, seed=5, field=qed.Field(B=(0.0, 0.0, 1e-3)), recoil_energy=recoil_energy)
        qed.run(tables, sp, p, 0, 1)
        qed.check(sp)
        out.append((qed.read_ledger(sp), [s.download() for s in sp]))
    (led, a), (_, b) = out
    assert led["emitted_n"] + led["dropped_n"] == few and led["pairs_n"] == few
    emitted = int(led["emitted_n"])
    for s, first, count in ((0, 0, few), (0, n, few), (1, 0, few), (2, 0, few), (2, n, emitted)):
        for key in ("x", "u", "tau", "id"):
            assert np.array_equal(a[s][key][first:first + count], b[s][key][first:first + count]), (s, first, key)
