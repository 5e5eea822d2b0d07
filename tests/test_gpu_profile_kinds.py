"""aew_profile_steps on the kernels that the solves run: two-step passes and on-chip runs, each
only where the handle has them, and a solve after them as before."""
import pytest
import torch

from paper_2304_04781_gb300 import inputs
from paper_2304_04781_gb300.aewave import AewError

from .helpers import cuda, setup, solver

pytestmark = pytest.mark.gpu

TWO = ["forward_two", "forward_pack_two", "adjoint_two", "adjoint_bf16_two", "incremental_bf16_two"]
CHIP = ["forward_chip", "adjoint_bf16_chip"]


@pytest.mark.parametrize("shape,kinds,route", [((160, 112, 112), TWO, "two"), ((32, 32, 32), CHIP, "chip")])
@pytest.mark.parametrize("nt", [32, 33])
def test_kinds_run_the_solves_kernels(shape, kinds, route, nt):
    prob, c, _ = setup(shape, nt, 16, seed=5)
    cc = cuda(c)
    s = solver(prob, storage="ae", codec="time")
    s.codec_set(inputs.codec_init(seed=4, n_hid=1024, n_lat=512))
    d_obs = torch.zeros((nt + 1, prob.nrec, 3), device="cuda")
    J, g = s.gradient(cc, d_obs)
    for kind in TWO + CHIP:
        if kind not in kinds:
            with pytest.raises(AewError, match="AEW_E_CONFIG"):
                s.profile(cc, kind, 3)
            continue
        a = s.routes()
        assert s.profile(cc, kind, 19) > 0
        b = s.routes()
        assert {k: b[k] - a[k] for k in b} == {"single": 0, "two": 0, "chip": 0, route: 19}
    J1, g1 = s.gradient(cc, d_obs)
    assert J1 == J and torch.equal(g1, g)


def test_kinds_need_the_time_codec():
    prob, c, _ = setup((32, 32, 32), 32, 16, seed=5)
    s = solver(prob)
    for kind in ("forward_pack_two", "adjoint_bf16_chip"):
        with pytest.raises(AewError, match="AEW_E_CONFIG"):
            s.profile(cuda(c), kind, 1)
    assert s.profile(cuda(c), "forward_chip", 3) > 0
