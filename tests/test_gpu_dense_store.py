"""Stored dense gradients at the edges of their blocks' columns and outputs, against the NumPy oracle."""
import numpy as np
import pytest

import oracle
from paper_2109_12191_b200 import synth
from gpu_util import TOL_FMA, TOL_NORM, gpu_layer, oracle_layer, rel_l2, scaled_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,Cin,Kout,bias", [(1, 1, 1, True), (3, 1028, 17, False), (2, 1023, 33, True), (5, 260, 1, True), (150, 12, 85, True),
                                             (20, 1024, 161, False)])
def test_dense_store(B, Cin, Kout, bias, dtype):
    layer = synth.dense(Cin, Kout, bias, "dense")
    inp = scaled_inputs(layer, B, dtype, 961, Cin, Kout, spread=True)
    dW, db = oracle_layer(layer, inp)
    out = gpu_layer(layer, inp, dtype, 0, bias_separate=0)
    assert rel_l2(out["G_w"], dW) <= TOL_FMA
    if bias:
        assert rel_l2(out["G_b"], db) <= TOL_FMA
    np.testing.assert_allclose(out["sq"][:, 0], oracle.sqnorm(dW) + (oracle.sqnorm(db) if bias else 0.0), rtol=TOL_NORM)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,Cin,Kout,bias", [(3, 644, 801, True), (130, 4740, 97, True), (1, 132, 2369, False), (2, 130, 2400, True)])
def test_dense_clipped_sum_of_a_large_output(B, Cin, Kout, bias, dtype):
    layer = synth.dense(Cin, Kout, bias, "dense")
    inp = scaled_inputs(layer, B, dtype, 962, Cin, Kout, spread=True)
    dW, db = oracle_layer(layer, inp)
    sq = oracle.sqnorm(dW) + (oracle.sqnorm(db) if bias else 0.0)
    C_l = float(np.sqrt(np.median(sq)))
    f = oracle.clip_factor(sq[:, None], C_l).reshape(B)
    out = gpu_layer(layer, inp, dtype, 2, bias_separate=0, C_l=C_l)
    assert rel_l2(out["acc_w"], np.einsum("n,np->p", f, dW)) <= TOL_FMA
    if bias:
        assert rel_l2(out["acc_b"], np.einsum("n,np->p", f, db)) <= TOL_FMA
