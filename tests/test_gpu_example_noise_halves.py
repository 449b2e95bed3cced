"""Per-example noise where half of the draws go with the norm pass: the fewest examples, odd counts, tensors on and off the
grid of Philox blocks in one call, and norms that are given, against the NumPy oracle."""
import math
import numpy as np
import pytest

from gpu_util import TOL_NORM
from test_gpu_example_noise import TOL_Z, _offsets, _oracle, _run, _spread

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Bn,sizes,first,given", [
    (7, [1028], 0, False), (8, [1028], 0, False), (9, [8196], 4, False), (257, [36], 0, False), (33, [1024, 9000, 3, 20], 4, False),
    (8, [4] * 530 + [2052, 5], 0, False), (11, [4096], 0, True),
    (9, [1025, 1023, 1, 2, 5, 1024], 3, False), (5, [2, 1021, 3], 1, False), (10, [1] * 600 + [1022], 2, False),
])
def test_noise_split_between_the_passes(Bn, sizes, first, given):
    groups, offs = _spread(Bn, sizes, Bn), _offsets(sizes, first)
    C, sigma, total = 0.3, 1.3, 4 * Bn
    acc0 = [np.linspace(-1, 1, p).astype(np.float32) for p in sizes]
    acc, norms, clip = _run("global", groups, offs, C, sigma, total, 22, 5, 3, acc0=acc0, give_norms=given)
    ref, sq, f = _oracle("global", groups, offs, C, sigma, total, 22, 5, 3, acc0=acc0)
    np.testing.assert_allclose(clip, f, rtol=TOL_NORM)
    sd = sigma * C / math.sqrt(total)
    for a, r in zip(acc, ref):
        assert np.max(np.abs(a - r)) <= Bn * sd * TOL_Z + 4e-6 * np.max(np.abs(r))
