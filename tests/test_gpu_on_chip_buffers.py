"""Buffers of the on-chip loops: made with the handle, not by its first solve."""
import pytest
import torch

from .helpers import cuda, setup, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(32, 32, 32), (64, 200, 36)])
def test_the_first_solve_allocates_nothing(shape):
    prob, c, _ = setup(shape, 20, 16, seed=5)
    cc = cuda(c)
    d_obs = torch.zeros((21, prob.nrec, 3), device="cuda")
    g, w = torch.empty_like(cc), cuda(c * 1e-3)
    x = torch.empty_like(cc)
    solver(prob).forward(cc)   # modules and streams are loaded by now
    s = solver(prob)
    held = s.stats()["device_bytes"]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s.forward(cc)
    s.gradient(cc, d_obs, g)
    s.hessvec(cc, x)
    torch.cuda.synchronize()
    assert s.routes()["chip"] > 0
    assert s.stats()["device_bytes"] == held and torch.cuda.mem_get_info()[0] == free
