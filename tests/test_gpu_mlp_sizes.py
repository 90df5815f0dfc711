"""Inference at the edges of its two kernels: one wave of 16-sample tiles (152 x 16 samples) and tiles of 128 beyond it.
Tolerance: FP32 sums of 128 terms over three layers, 1e-5 of the largest output (as for the other kernels' test)."""
import numpy as np
import pytest

import synth
from oracle import mlp
from tests.gpu_util import context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 17, 2432, 2433, 128 * 152 + 1, 20001])
def test_predict_sizes(n):
    ctx = context()
    try:
        ctx.mlp_set_params(synth.mlp_init(15))
        _, comp = ctx.mlp_get_params()
        X = np.random.default_rng(n).standard_normal((n, 6)).astype(np.float32)
        mu, lv = ctx.mlp_predict(X)
    finally:
        ctx.close()
    out, _ = mlp.forward(comp.astype(float), X.astype(float))
    assert np.max(np.abs(mu - out[:, 0])) <= 1e-5 * np.max(np.abs(out[:, 0]))
    assert np.max(np.abs(lv - out[:, 1])) <= 1e-5 * np.max(np.abs(out[:, 1]))
