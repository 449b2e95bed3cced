"""Image stems (3x3 filters on three channels): the blocks of an example's cluster against the NumPy oracle."""
import numpy as np
import pytest

import oracle
from paper_2109_12191_b200 import synth
from gpu_util import TOL_FMA, TOL_NORM, gpu_layer, oracle_layer, rel_l2, scaled_inputs

pytestmark = pytest.mark.gpu

STORE, NORM = 0, 1

CASES = [
    # B, Kout, stride, pad, H, W, bias: how the output rows fall to the blocks
    (2, 32, 1, 1, 15, 17, True),        # 255 pixels: one block
    (2, 32, 1, 1, 16, 17, True),        # 272: two blocks of eight rows
    (3, 32, 1, 0, 37, 41, True),        # eight blocks of five rows, the last one without any
    (3, 32, 2, 1, 57, 25, False),       # stride 2
    (160, 32, 1, 1, 38, 40, True),      # more examples than SMs: one block each
    (90, 64, 2, 1, 25, 13, False),      # 64 channels: the ring is reused
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("case", CASES)
def test_stem_conv_over_a_cluster_of_blocks(case, dtype):
    B, Kout, stride, pad, H, W, bias = case
    layer = synth.Layer("conv", 3, Kout, R=3, S=3, stride=stride, pad=pad, H=H, W=W, bias=bias, name=str(case))
    inp = scaled_inputs(layer, B, dtype, 951, B, H, spread=True)
    dW, db = oracle_layer(layer, inp)
    groups = 2 if bias else 1
    sq = np.stack([oracle.sqnorm(dW), oracle.sqnorm(db)], 1) if bias else oracle.sqnorm(dW)[:, None]
    out = gpu_layer(layer, inp, dtype, STORE, bias_separate=groups - 1)
    for n in range(B):
        assert rel_l2(out["G_w"][n], dW[n]) <= TOL_FMA
        if bias:
            assert rel_l2(out["G_b"][n], db[n]) <= TOL_FMA
    np.testing.assert_allclose(out["sq"], sq, rtol=TOL_NORM)
    out = gpu_layer(layer, inp, dtype, NORM)
    np.testing.assert_allclose(out["sq"], sq.sum(1, keepdims=True), rtol=TOL_NORM)
