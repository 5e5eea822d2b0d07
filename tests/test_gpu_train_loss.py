"""The training loss is an FP64 sum: finite where a square overflows FP32, and complete where
squares lie below FP32's normal range."""
import numpy as np
import pytest
import torch

from paper_2304_04781_gb300 import inputs

from .helpers import setup, solver

pytestmark = pytest.mark.gpu


def loss_of(b4, batch, codec):
    """Loss of one minibatch of zeros under a decoder that returns b4 whatever it reads."""
    prob, _, _ = setup((16, 16, 16), 2, 4)
    s = solver(prob, codec=codec)
    W = inputs.codec_init(seed=4, n_hid=s.n_hid, n_lat=s.n_lat)
    W["W4"] = np.zeros_like(W["W4"])
    W["b4"] = b4.astype(np.float32)
    s.codec_set(W)
    Y = torch.zeros((batch, 2048), device="cuda", dtype=torch.bfloat16)
    return s.codec_train(Y, epochs=1, batch=batch, lr0=0.0)[0]


@pytest.mark.parametrize("codec", ["time", "space"])
@pytest.mark.parametrize("scale", [1.0, 5e19, 1e-24])
@pytest.mark.parametrize("batch", [8, 136])
def test_loss_is_an_fp64_sum(codec, scale, batch):
    """Every term is exact in FP64 (squares of FP32 values).  A sum of n terms is off by
    (n - 1) 2^-53 at most: 32 per lane, 5 across a warp, one per warp of rows and column
    group, and the divisions."""
    b4 = (np.random.default_rng(1).standard_normal(2048) * scale).astype(np.float32)
    want = np.mean(b4.astype(np.float64) ** 2)
    got = loss_of(b4, batch, codec)
    n = 32 + 5 + 64 * ((batch + 31) // 32) + 4
    assert abs(got - want) <= n * 2.0 ** -53 * want, (got, want)
