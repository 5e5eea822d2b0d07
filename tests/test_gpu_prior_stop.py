"""Where the streaming prior solve stops: the launches enqueued past the passing residual test
(one with the test itself, then plain ones) leave x and the iteration count as they were."""
import numpy as np
import pytest

from paper_2304_04781_gb300 import inputs

from .helpers import cuda, host, setup, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(8, 12, 132), (40, 52, 64), (64, 96, 128)])
@pytest.mark.parametrize("rtol", [1e-2, 1e-6])
def test_launches_past_the_passing_test_change_nothing(shape, rtol, monkeypatch):
    monkeypatch.setenv("AEW_STENCIL_KC_FWD", "8")   # the streaming kernels on every grid
    prob, _, _ = setup(shape, 4, 4)
    s = solver(prob, storage="full")
    w = cuda(inputs.white_noise(1, prob.shape, seed=6)[0])
    theta = 2.0 * prob.h ** 2
    x, it = s.prior_solve(w, 0.5, theta, rtol=rtol)
    assert it % 8 == 0 and it > 0
    for _ in range(20):
        y, again = s.prior_solve(w, 0.5, theta, rtol=rtol)
        assert again == it and np.array_equal(host(y), host(x))
    # the last iteration allowed: nothing is enqueued past it
    y, again = s.prior_solve(w, 0.5, theta, rtol=rtol, max_iter=it)
    assert again == it and np.array_equal(host(y), host(x))
