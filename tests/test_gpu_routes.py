"""Which kernels run the time steps: on-chip runs and two-step passes only where they are
the faster ones (the lines and both sides' times stand at the rules)."""
import numpy as np
import pytest
import torch

from paper_2304_04781_gb300 import inputs

from .helpers import cuda, setup, solver

pytestmark = pytest.mark.gpu


def routes_of(s, run):
    """Launches of (single steps, two-step passes, on-chip runs) made by run()."""
    a = s.routes()
    run()
    b = s.routes()
    return tuple(b[k] - a[k] for k in ("single", "two", "chip"))


@pytest.mark.parametrize("shape", [(32, 32, 32), (96, 96, 96)])
def test_space_codec_steps_beside_the_codec_are_single(shape):
    """A cooperative launch would wait for the decoder beside it to leave it all its SMs."""
    nt = 6
    prob, c, _ = setup(shape, nt, 16, seed=5)
    cc, dc = cuda(c), cuda(np.ones(shape))
    d_obs = torch.zeros((nt + 1, prob.nrec, 3), device="cuda")
    s = solver(prob, storage="ae")
    s.codec_set(inputs.codec_init(seed=4))
    assert routes_of(s, lambda: s.gradient(cc, d_obs)) == (2 * nt, 0, 0)
    assert routes_of(s, lambda: s.hessvec(dc)) == (2 * nt, 0, 0)


def test_space_codec_leaves_half_the_gpu_to_the_step_beside_it(monkeypatch):
    """Its solves run single steps on every grid, so its decoder is capped at half the SMs
    there too: 256 tiles take four rounds on 76 CTAs, two on 152."""
    shape = (256, 256, 256)
    prob, c, _ = setup(shape, 2, 4, seed=5)
    cc = cuda(c)

    def decode_ms(cap):
        monkeypatch.delenv("AEW_GEMM_CTAS_OVERLAP", raising=False)
        if cap is not None:
            monkeypatch.setenv("AEW_GEMM_CTAS_OVERLAP", cap)
        s = solver(prob, storage="ae")
        s.codec_set(inputs.codec_init(seed=4))
        s.profile(cc, "decode_state", 5)
        ms = s.profile(cc, "decode_state", 50)
        s.close()
        return ms

    free, capped = decode_ms("0"), decode_ms(None)
    assert 1.4 * free < capped < 3.0 * free, (free, capped)


@pytest.mark.parametrize("shape,chip", [((32, 32, 32), True), ((104, 104, 104), True),
                                        ((112, 112, 112), False), ((24, 256, 256), False)])
def test_single_steps_go_on_chip_on_small_bricks_only(shape, chip):
    """The JVP with checkpoints runs forward and incremental steps in turn, and data of every
    state ends a run at each: runs of one step.  Runs of two and more stay on chip."""
    nt = 9
    prob, c, _ = setup(shape, nt, 16, seed=5)
    cc, dc = cuda(c), cuda(np.ones(shape))
    s = solver(prob, storage="revolve", n_checkpoints=2)
    s.gradient(cc, torch.zeros((nt + 1, prob.nrec, 3), device="cuda"))
    n = 2 * nt - 1
    assert routes_of(s, lambda: s.jvp(dc)) == ((0, 0, n) if chip else (n, 0, 0))
    room = nt * s.nblocks
    one, _, many = routes_of(s, lambda: s.snapshots(cc, 1, room))
    assert (one == 0 and many == nt - 1) if chip else (one >= nt - 1 and many == 0)
    assert routes_of(s, lambda: s.snapshots(cc, 2, room)) == (0, 0, (nt - 1) // 2)


@pytest.mark.parametrize("shape,least", [((20, 24, 28), 1), ((112, 112, 112), 3)])
@pytest.mark.parametrize("nsteps", [1, 2, 3, 4, 8])
def test_propagate_routes_and_bits(shape, least, nsteps, monkeypatch):
    """On chip from `least` steps on, two launches that end in the caller's buffers; the same
    bits as the streaming kernels either way."""
    prob, c, _ = setup(shape, 10, 16, seed=5)
    cc, rng = cuda(c), np.random.default_rng(3)
    state = [cuda(rng.standard_normal(shape)) for _ in range(4)]
    wav = rng.standard_normal(nsteps).astype(np.float32)
    out = []
    for kc in (None, "6"):
        if kc:
            monkeypatch.setenv("AEW_STENCIL_KC_FWD", kc)   # the streaming kernels
        s = solver(prob)
        for w in (None, wav):
            st = [x.clone() for x in state]
            rec = []
            n = routes_of(s, lambda: rec.append(s.propagate(cc, st, 0, nsteps, wavelet=w, record=True)))
            chip = not kc and nsteps >= least
            assert n == ((0, 0, min(nsteps, 2)) if chip else (nsteps, 0, 0))
            out.append([rec[0], *st])
        s.close()
    for a, b in zip(out[:2], out[2:]):
        assert all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("shape,plain", [((8, 512, 512), False), ((4, 64, 4096), False),
                                         ((64, 64, 512), True), ((100, 104, 260), True),
                                         ((24, 256, 512), True), ((160, 112, 112), True)])
def test_two_steps_per_pass_where_they_are_faster(shape, plain, monkeypatch):
    """Grids beyond the SMs: single forward and adjoint steps where x needs several tiles,
    rows are whole tiles of the single-step kernels and the state stays in L2; the same bits
    as with single steps everywhere."""
    nt = 6
    prob, c, _ = setup(shape, nt, 1, seed=5)
    cc, rng = cuda(c), np.random.default_rng(3)
    d_obs = cuda(rng.standard_normal((nt + 1, prob.nrec, 3)) * 1e-6)
    dc = cuda(rng.standard_normal(shape))
    out = []
    for kc in (None, "6"):
        if kc:
            monkeypatch.setenv("AEW_STENCIL_KC_FWD", kc)   # single steps
        s = solver(prob)
        res = []

        def run():
            res.extend([s.forward(cc), *s.gradient(cc, d_obs)[::-1], s.hessvec(dc)])

        n = routes_of(s, run)
        if kc:
            assert n == (5 * nt, 0, 0)
        else:
            assert n == ((0, 5 * nt // 2, 0) if plain else (4 * nt, nt // 2, 0))
        out.append(res)
        s.close()
    for a, b in zip(*out):
        assert torch.equal(a, b) if isinstance(a, torch.Tensor) else a == b
