"""The on-chip prior solve in several launches: how many iterations a launch takes changes no bit,
and a large max_iter is not one launch."""
import numpy as np
import pytest

from oracle import newton as NW
from paper_2304_04781_gb300 import inputs
from paper_2304_04781_gb300.aewave import AewError

from .helpers import cuda, host, relerr, setup, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 12, 20), (60, 36, 44), (96, 96, 96), (112, 112, 128)])
def test_iterations_per_launch_change_no_bit(shape, monkeypatch):
    prob, _, _ = setup(shape, 4, 4)
    s = solver(prob)
    w = cuda(inputs.white_noise(1, prob.shape, seed=6)[0])
    theta = 64.0 * prob.h ** 2
    out = []
    for run in (None, "8", "24"):
        if run:
            monkeypatch.setenv("AEW_PRIOR_RUN", run)
        x, it = s.prior_solve(w, 0.5, theta, rtol=1e-5)
        out.append((it, host(x)))
        with pytest.raises(AewError, match="NOCONVERGE"):   # not a multiple of 8, x is the last iterate
            s.prior_solve(w, 0.5, theta, rtol=1e-12, max_iter=29, out=x)
        out[-1] += (host(x),)
    for o in out[1:]:
        assert o[0] == out[0][0] > 24 and np.array_equal(o[1], out[0][1]) and np.array_equal(o[2], out[0][2])


def test_more_iterations_than_a_launch_takes():
    """A condition number of 1.2e6 on a long grid: over a thousand iterations.  The recursive
    residual meets the tolerance; FP32 rounding adds eps |A| |x| to the true one per iteration."""
    prob, _, _ = setup((16, 32, 512), 4, 4)
    s = solver(prob)
    w = inputs.white_noise(1, prob.shape, seed=6)[0].astype(np.float32).astype(np.float64)
    theta = 1e5 * prob.h ** 2
    x, it = s.prior_solve(cuda(w), 0.5, theta, rtol=1e-5, max_iter=100000)
    assert it > 1024
    scale = 0.5 * (1 + 12 * theta / prob.h ** 2) * np.linalg.norm(host(x)) / np.linalg.norm(w)
    res = relerr(NW.prior_apply(host(x), prob.h, 0.5, theta), w)
    assert res <= 1e-5 + 2 * np.sqrt(it) * 2.0 ** -24 * scale, (it, res, scale)
