"""The prior solve over grids that cut its tiles everywhere: x in one, two and three tiles of
128 nodes, rows in one and more blocks of ten, planes in chunks, the smallest grid."""
import numpy as np
import pytest

from oracle import newton as NW
from paper_2304_04781_gb300 import inputs

from .helpers import cuda, host, relerr, setup, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("streaming", [False, True])
@pytest.mark.parametrize("shape", [(4, 4, 4), (4, 12, 132), (12, 40, 128), (12, 24, 260), (68, 12, 8), (40, 52, 64)])
def test_prior_solve_residual(shape, streaming, monkeypatch):
    """theta = 2 h^2: condition number 25.  FP32 rounding adds eps |A| |x| <= 25 eps |w| to the
    residual per iteration, independent from one to the next: 2 sqrt(it) 25 eps on top of rtol."""
    if streaming:
        monkeypatch.setenv("AEW_STENCIL_KC_FWD", "8")
    prob, _, _ = setup(shape, 4, 4)
    s = solver(prob, storage="full")
    w = inputs.white_noise(1, prob.shape, seed=6)[0].astype(np.float32).astype(np.float64)
    theta = 2.0 * prob.h ** 2
    x, it = s.prior_solve(cuda(w), 0.5, theta, rtol=1e-6)
    res = relerr(NW.prior_apply(host(x), prob.h, 0.5, theta), w)
    assert it % 8 == 0 and res <= 1e-6 + 2 * np.sqrt(it) * 25 * 2.0 ** -24
    with pytest.raises(Exception):
        s.prior_solve(cuda(w), 0.5, theta, rtol=1e-6, max_iter=3 if it > 8 else 1)
    # and the handle still solves
    assert np.array_equal(host(s.prior_solve(cuda(w), 0.5, theta, rtol=1e-6)[0]), host(x))
