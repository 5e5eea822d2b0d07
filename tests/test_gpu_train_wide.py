"""A training step on a batch wide enough for 256-column tiles (every SM has one), with a ragged
last tile of rows, against the oracle's LAMB step."""
import numpy as np
import pytest
import torch

from oracle import codec as C
from paper_2304_04781_gb300 import inputs

from .helpers import relerr, setup, solver

pytestmark = pytest.mark.gpu


def test_wide_batch_step_equals_the_oracle():
    """The tolerances of the batch-256 test against the same oracle: BF16 operands, 2e-3 on the
    weights and 1e-2 on the inner biases, whose near-zero gradient entries LAMB's first, nearly
    sign-like step may move the other way."""
    n = 2440   # 20 row tiles x 8 column tiles of 256 on 152 SMs, 8 rows in the last
    prob, _, _ = setup((32, 32, 32), 4, 16)
    s = solver(prob, storage="full", codec="time", n_lat=512)
    Wt = inputs.codec_init(seed=5, n_hid=s.n_hid, n_lat=512)
    s.codec_set(Wt)
    rng = np.random.default_rng(6)
    Y = C.round_bf16(rng.uniform(-1, 1, (n, 2048)) * rng.uniform(0.05, 1.0, (n, 1)))
    loss = s.train_step(torch.from_numpy(Y.astype(np.float32)).to(torch.bfloat16).cuda(), 1e-3)
    Wo = {k: v.astype(np.float64) for k, v in Wt.items()}
    L, g = C.loss_and_grad(Wo, Y, emulate=True)
    assert abs(loss - L) <= 2e-3 * L
    Wo = C.Lamb(Wo).step(Wo, g, 1e-3)
    Wg = s.codec_get()
    for k in C.PARAMS:
        assert relerr(Wg[k], Wo[k]) < (1e-2 if k in ("b1", "b2", "b3") else 2e-3), k
