"""Two steps per pass (grids too large for the on-chip loops) against single streaming steps,
bit for bit: x in one, two, three and more tiles, partial last tiles, columns and z chunks,
odd and even step counts, receivers and the source on tile edges."""
import numpy as np
import pytest
import torch

from oracle import wave as W
from paper_2304_04781_gb300 import inputs
from tests.helpers import cuda, setup, solver
from tests.test_gpu_brick import both, same

pytestmark = pytest.mark.gpu

SHAPES = [(160, 112, 112), (132, 132, 132), (100, 104, 260), (12, 16, 600), (4, 8, 2052), (20, 36, 1032),
          (1040, 100, 24)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("nt", [9, 12])
def test_solves_equal_single_steps(shape, nt, monkeypatch):
    prob, c, _ = setup(shape, nt, 16, seed=5)
    cc, rng = cuda(c), np.random.default_rng(3)
    state = [cuda(rng.standard_normal(shape)) for _ in range(4)]
    wav = rng.standard_normal(nt).astype(np.float32)
    d_obs = cuda(rng.standard_normal((nt + 1, prob.nrec, 3)) * 1e-6)
    dc = cuda(rng.standard_normal(shape))

    def run(s):
        st = [x.clone() for x in state]
        rec = s.propagate(cc, st, 0, nt, wavelet=wav, record=True)
        J, g = s.gradient(cc, d_obs)
        out = [s.forward(cc), s.forward(cc, wavelet=wav), rec, *st, g, J]
        s.gradient(cc, d_obs)
        out += [s.hessvec(dc), s.jvp(dc)]
        if s.stats()["history_bytes"] == nt * c.size * 4:
            out.append(s.hessvec_full(dc))
        return out

    for kw in ({}, {"storage": "revolve", "n_checkpoints": 2}, {"accum_window": 1}, {"accum_window": 3}):
        same(*both(monkeypatch, lambda: solver(prob, **kw), run))


@pytest.mark.parametrize("shape,nt", [((160, 112, 112), 33), ((132, 136, 136), 36), ((100, 104, 264), 17),
                                      ((20, 40, 1032), 35), ((1040, 104, 24), 18)])
@pytest.mark.parametrize("norm", ["pow2", "minmax"])
def test_time_codec_equals_single_steps(shape, nt, norm, monkeypatch):
    """Window packing across window boundaries, the maxima, and the BF16 reads."""
    prob, c, _ = setup(shape, nt, 16, seed=6)
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


def test_source_and_receivers_on_tile_edges(monkeypatch):
    """A smoothed source over an x tile boundary and over column and chunk edges, receivers on
    every node of a row and on the first and last planes' neighbours."""
    shape = (96, 112, 264)
    for k in (1, 48, 94):
        rec = np.array([(i, 57, k) for i in range(1, 263, 5)], np.int32)
        prob = W.Problem(shape=shape, h=10.0, nt=8, rec=rec, src_sigma=30.0)
        c = inputs.velocity_model(shape, 10.0, seed=7).astype(np.float32)
        d_obs = torch.ones((9, len(rec), 3), device="cuda") * 1e-6
        same(*both(monkeypatch, lambda: solver(prob),
                   lambda s: [s.forward(cuda(c)), *s.gradient(cuda(c), d_obs)]))
