"""The on-chip time loops (grids that fit the SMs) against the streaming kernels, bit for
bit: both evaluate the same expressions, so any difference is an error of the cut, the
halo exchange or the launch's bookkeeping.  A z-chunk depth set by hand makes a handle use
the streaming kernels."""
import numpy as np
import pytest
import torch

from oracle import wave as W
from paper_2304_04781_gb300 import inputs
from tests.helpers import cuda, setup, solver

pytestmark = pytest.mark.gpu

# one node column per brick, short and long rows (x rows across warps), partial last bricks,
# every brick depth, a brick per SM
SHAPES = [(4, 4, 4), (8, 12, 20), (32, 32, 32), (60, 36, 44), (16, 8, 256), (152, 8, 16),
          (72, 100, 148), (64, 200, 36), (100, 96, 96), (112, 112, 128), (128, 128, 128),
          (100, 60, 252), (20, 52, 480)]


def both(monkeypatch, make, run):
    """run(solver) with the on-chip loops and with the streaming kernels."""
    out = []
    for kc in (None, "6"):
        if kc is None:
            monkeypatch.delenv("AEW_STENCIL_KC_FWD", raising=False)
        else:
            monkeypatch.setenv("AEW_STENCIL_KC_FWD", kc)   # read when the handle is made
        s = make()
        out.append(run(s))
        s.close()
    return out


def same(a, b):
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert torch.equal(x, y) if isinstance(x, torch.Tensor) else x == y


@pytest.mark.parametrize("shape", SHAPES)
def test_solves_equal_the_streaming_kernels(shape, monkeypatch):
    """Seismograms (default and given wavelet), a propagated state, gradients and GN-HVPs
    with full storage and with checkpoints (segments of many and of single steps), and the
    full Newton HVP; 21 steps (two accumulation windows and a part)."""
    prob, c, _ = setup(shape, 21, 16 if min(shape[1:]) >= 8 else 1, seed=5)
    cc = cuda(c)
    rng = np.random.default_rng(3)
    state = [cuda(rng.standard_normal(shape)) for _ in range(4)]
    wav = rng.standard_normal(21).astype(np.float32)
    d_obs = cuda(rng.standard_normal((22, prob.nrec, 3)) * 1e-6)
    dc = cuda(rng.standard_normal(shape))

    def run(s):
        st = [x.clone() for x in state]
        rec = s.propagate(cc, st, 0, 9, wavelet=wav[:9], record=True)
        J, g = s.gradient(cc, d_obs)
        out = [s.forward(cc), s.forward(cc, wavelet=wav), rec, *st, g, J]
        J, g = s.gradient(cc, d_obs)
        out += [s.hessvec(dc), s.jvp(dc)]
        if s.stats()["history_bytes"] == 21 * c.size * 4:
            out.append(s.hessvec_full(dc))
        return out

    for kw in ({}, {"storage": "revolve", "n_checkpoints": 3}):
        same(*both(monkeypatch, lambda: solver(prob, **kw), run))


@pytest.mark.parametrize("shape,nt", [((8, 8, 8), 1), ((32, 32, 32), 16), ((36, 40, 104), 17),
                                      ((96, 96, 96), 37), ((128, 128, 128), 35)])
@pytest.mark.parametrize("norm", ["pow2", "minmax"])
def test_time_codec_equals_the_streaming_kernels(shape, nt, norm, monkeypatch):
    """Window packing, the window maxima and the BF16 reads: gradient, GN-HVP, JVP and full
    Newton HVP with the time codec, window counts with and without a partial last window."""
    prob, c, _ = setup(shape, nt, 1 if shape[1] == 8 else 16, seed=6)
    cc, rng = cuda(c), np.random.default_rng(4)
    d_obs = cuda(rng.standard_normal((nt + 1, prob.nrec, 3)) * 1e-6)
    dc = cuda(rng.standard_normal(shape))
    Wt = inputs.codec_init(seed=4, n_hid=1024, n_lat=512)

    def make():
        s = solver(prob, storage="ae", codec="time", norm=norm)
        s.codec_set(Wt)
        return s

    def run(s):
        J, g = s.gradient(cc, d_obs)
        return [J, g, s.hessvec(dc), s.jvp(dc), s.hessvec_full(dc)]

    same(*both(monkeypatch, make, run))


@pytest.mark.parametrize("codec,every,room", [("space", 1, 4), ("space", 7, 99), ("time", 1, 99),
                                              ("time", 2, 99)])
@pytest.mark.parametrize("shape", [(8, 8, 8), (24, 40, 72), (96, 96, 96)])
def test_snapshots_equal_the_streaming_kernels(shape, codec, every, room, monkeypatch):
    """Algorithm 1: packed vectors and maxima, with room for some or all of the states."""
    prob, c, _ = setup(shape, 67, 1, seed=9)

    def run(s):
        unit = s.nvec if codec == "time" else s.nblocks
        v, m = s.snapshots(cuda(c), every, room * unit + 1, with_scales=True)
        return [v, m, s.snapshots(cuda(c), every, room * unit)]

    same(*both(monkeypatch, lambda: solver(prob, storage="revolve", n_checkpoints=0, codec=codec), run))


def test_smoothed_source_and_window_of_one(monkeypatch):
    """A source spread over many bricks, and an FP64 flush in every step."""
    shape = (48, 52, 56)
    prob = W.Problem(shape=shape, h=10.0, nt=30, rec=inputs.receiver_grid(56, 52, 16), src_sigma=50.0)
    c = inputs.velocity_model(shape, 10.0, seed=7).astype(np.float32)
    d_obs = torch.zeros((31, 16, 3), device="cuda")
    for aw in (1, 40):
        same(*both(monkeypatch, lambda: solver(prob, accum_window=aw),
                   lambda s: [s.forward(cuda(c)), *s.gradient(cuda(c), d_obs)]))


def test_a_given_up_wait_is_reported_and_the_handle_recovers():
    """A set error flag: the on-chip kernels return at once, the next synchronising call
    reports it, and the results after it are those of a fresh handle."""
    from paper_2304_04781_gb300.aewave import AewError
    prob, c, _ = setup((32, 32, 32), 40, 16, seed=8)
    d_obs = torch.zeros((41, 16, 3), device="cuda")
    s, ref = solver(prob), solver(prob)
    s.test_wait_timeout(1_000_000)
    s.forward(cuda(c))
    with pytest.raises(AewError, match="AEW_E_TIMEOUT"):
        s.sync_check()
    same([*s.gradient(cuda(c), d_obs)], [*ref.gradient(cuda(c), d_obs)])
