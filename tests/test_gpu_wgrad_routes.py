"""Forms of single weight-gradient calls that only some sizes take, each test making sure that its call takes the form."""
import numpy as np
import pytest
import torch

import oracle
from paper_2109_12191_b200 import synth
from gpu_util import B, TOL_FMA, TOL_NORM, dev_inputs, kernels_of, make_desc, oracle_layer, rel_l2, scaled_inputs

pytestmark = pytest.mark.gpu

STORE, NORM, CLIP = 0, 1, 2


class Call:
    """One layer call and its buffers; filled with a value that the library does not write."""

    def __init__(self, layer, Bn, dtype, epi, key):
        b = B()
        self.inp = scaled_inputs(layer, Bn, dtype, key, Bn)
        self.epi, self.desc, self.data = epi, make_desc(layer, Bn, dtype), dev_inputs(self.inp, dtype)
        self.G = torch.full((Bn, layer.n_weight), -7.0, device="cuda") if epi == STORE else None
        self.acc = torch.zeros(layer.n_weight, device="cuda") if epi == CLIP else None
        self.sq, self.clip = (torch.full((Bn, 1), -7.0, device="cuda") for _ in range(2))
        self.ws = torch.empty(b.dp_workspace_bytes(self.desc, epi), dtype=torch.uint8, device="cuda")
        b.check(b.dp_workspace_init(self.ws))
        self.dW, _ = oracle_layer(layer, self.inp)
        self.C_l = float(np.sqrt(np.median(oracle.sqnorm(self.dW))))

    def __call__(self):
        b = B()
        b.check(b.dp_per_example_wgrad(self.desc, *self.data, self.G, None, self.sq, 1, self.epi, self.C_l, self.acc, None,
                                       self.clip if self.epi == CLIP else None, self.ws))

    def times_out(self):
        """Runs with waits that give up at once, then again on the same workspace: the first is reported, the second is right."""
        b = B()
        b.dp_debug_set_wait_polls(0)
        try:
            self()
            torch.cuda.synchronize()
        finally:
            b.dp_debug_set_wait_polls(-1)
        left = [t.clone() for t in (self.sq, self.clip, self.G, self.acc) if t is not None]
        assert b.dp_wgrad_check(self.ws) == b.DP_ERR_TIMEOUT
        if self.acc is not None:
            self.acc.zero_()
        self()
        b.check(b.dp_wgrad_check(self.ws))
        self.is_right()
        return left

    def is_right(self):
        sq = oracle.sqnorm(self.dW)
        np.testing.assert_allclose(self.sq.cpu().numpy()[:, 0], sq, rtol=TOL_NORM)
        if self.epi == STORE:
            assert rel_l2(self.G.cpu().numpy(), self.dW) <= TOL_FMA
        if self.epi == CLIP:
            f = oracle.clip_factor(sq, self.C_l)
            np.testing.assert_allclose(self.clip.cpu().numpy()[:, 0], f, rtol=TOL_NORM)
            assert rel_l2(self.acc.cpu().numpy(), np.einsum("n,np->p", f, self.dW)) <= TOL_FMA


@pytest.mark.parametrize("layer,Bn", [(synth.conv(64, 64, 1, 1, 0, 50), 1), (synth.conv(64, 256, 1, 1, 0, 37), 3), (synth.conv(3, 64, 7, 2, 3, 96), 2)])
@pytest.mark.parametrize("epi", [STORE, NORM])
def test_pixels_shared_by_a_cluster_with_waits_that_give_up(layer, Bn, epi):
    """No squared norm is made of tiles that were never written, and none of the stored gradients either."""
    call = Call(layer, Bn, "bf16", epi, 982)
    call()                                                   # (whatever a first call sets up, outside the capture)
    torch.cuda.synchronize()
    assert any("conv_wgrad_split_kernel" in name for name in kernels_of(call))
    call.sq.fill_(-7.0)
    if call.G is not None:
        call.G.fill_(-7.0)
    sq, _, *G = call.times_out()
    assert bool(torch.isnan(sq).all())
    assert all(bool((g == -7.0).all()) for g in G)


GRAM_CONVS = [
    # gradients too large for a cluster, output planes of at most 256 pixels: two row tiles, the second with 96 rows, with 16; one row
    # tile, mostly zero rows; strided taps; strided 1 x 1; flattened pixels, 196 -> 208 rows; exactly 256 pixels
    synth.conv(128, 256, 3, 1, 1, 14), synth.conv(128, 256, 3, 1, 1, 10), synth.conv(128, 256, 3, 1, 1, 5), synth.conv(128, 256, 3, 2, 1, 14),
    synth.conv(512, 1024, 1, 2, 0, 14), synth.conv(1024, 512, 1, 1, 0, 14), synth.conv(256, 1152, 1, 1, 0, 16),
]


@pytest.fixture
def side_by_side():
    b = B()
    b.check(b.dp_set_sm_target(torch.cuda.get_device_properties(0).multi_processor_count))
    yield
    b.check(b.dp_set_sm_target(0))


@pytest.mark.parametrize("layer", GRAM_CONVS)
def test_norms_from_gram_matrices_side_by_side(layer, side_by_side):
    """Calls that run side by side with others take their norms from the Gram matrices of the pixels."""
    call = Call(layer, 5, "bf16", CLIP, 983)
    call()
    call.is_right()
    assert any("conv_gram_norm_kernel" in name for name in kernels_of(call))


def test_gram_matrices_with_waits_that_give_up(side_by_side):
    call = Call(GRAM_CONVS[0], 3, "bf16", CLIP, 984)
    call()
    torch.cuda.synchronize()
    assert any("conv_gram_norm_kernel" in name for name in kernels_of(call))
    call.times_out()


@pytest.mark.parametrize("Bn,gram", [(10, False), (11, True)])
def test_norms_of_very_many_tiles_over_few_pixels(Bn, gram):
    """512 x 4608 entries an example over 25 pixels: by tiles up to 24 million of them, from Gram matrices past that."""
    call = Call(synth.conv(512, 512, 3, 1, 1, 5), Bn, "bf16", CLIP, 985)
    call()
    call.is_right()
    assert any("conv_gram_norm_kernel" in name for name in kernels_of(call)) == gram
