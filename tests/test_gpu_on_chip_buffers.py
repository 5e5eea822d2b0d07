"""Buffers of the on-chip loops: made with the handle, not by its first solve."""
import numpy as np
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


def test_a_given_wavelet_allocates_nothing():
    """forward and propagate with a caller's wavelet, also one longer than the handle's nt."""
    shape, nt = (32, 32, 32), 20
    prob, c, _ = setup(shape, nt, 16, seed=5)
    s, cc = solver(prob), cuda(c)
    held = s.stats()["device_bytes"]
    wav = np.ones(3 * nt, np.float32)
    s.forward(cc, wavelet=wav[:nt])
    s.propagate(cc, [torch.zeros_like(cc) for _ in range(4)], 0, 3 * nt, wavelet=wav)
    assert s.routes()["single"] == 0 and s.stats()["device_bytes"] == held


@pytest.mark.parametrize("nt,nsteps", [(1, 1), (1, 3), (3, 7), (5, 26), (1000, 1999)])
def test_a_wavelet_longer_than_its_buffer(nt, nsteps, monkeypatch):
    """propagate takes more steps than the handle's nt: in parts, the same bits as streaming;
    1000 values and more also fill several argument chunks."""
    shape = (8, 12, 20)
    prob, c, _ = setup(shape, nt, 1, seed=5)
    cc, rng = cuda(c), np.random.default_rng(3)
    state = [cuda(rng.standard_normal(shape)) for _ in range(4)]
    wav = rng.standard_normal(nsteps).astype(np.float32)
    out = []
    for kc in (None, "6"):
        if kc:
            monkeypatch.setenv("AEW_STENCIL_KC_FWD", kc)   # the streaming kernels
        s = solver(prob)
        st = [x.clone() for x in state]
        out.append([s.propagate(cc, st, 0, nsteps, wavelet=wav, record=True), *st,
                    s.forward(cc, wavelet=wav[:nt])])
    assert all(torch.equal(x, y) for x, y in zip(*out))
