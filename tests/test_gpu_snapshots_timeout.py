"""Data generation after a bounded wait that gave up: the step kernels return at once, so the
packed vectors are void.  The call says so, and the handle's next call is right again."""
import pytest
import torch

from .helpers import cuda, setup, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("codec", ["space", "time"])
@pytest.mark.parametrize("streaming", [False, True])
def test_snapshots_report_a_given_up_wait(codec, streaming, monkeypatch):
    from paper_2304_04781_gb300.aewave import AewError
    if streaming:
        monkeypatch.setenv("AEW_STENCIL_KC_FWD", "6")
    prob, c, _ = setup((32, 32, 32), 40, 16, seed=8)
    s, ref = (solver(prob, storage="revolve", n_checkpoints=0, codec=codec) for _ in range(2))
    room = 99 * (s.nvec if codec == "time" else s.nblocks)
    s.test_wait_timeout(1_000_000)
    with pytest.raises(AewError, match="AEW_E_TIMEOUT"):
        s.snapshots(cuda(c), 1, room)
    (v, m), (v0, m0) = (x.snapshots(cuda(c), 1, room, with_scales=True) for x in (s, ref))
    assert v.shape[0] > 0 and torch.equal(v, v0) and torch.equal(m, m0)
