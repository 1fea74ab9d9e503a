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
