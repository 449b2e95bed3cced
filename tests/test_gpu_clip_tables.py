"""Clipping at the edges of its launches: rows at any address, blocks that share rows, large tensors and many tensors,
against the NumPy oracle."""
import pytest

from test_gpu_clip import _check, _spread

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("give_norms", [False, True])
@pytest.mark.parametrize("sizes,Bn", [
    ([1031], 15), ([1031], 16),           # the fewest rows whose warps share a block, and one less; unaligned rows
    ([129, 3, 4100], 17),                 # one column past a narrow block; aligned and unaligned tensors in one launch
    ([127], 300),                         # more rows than one round of factors
    ([8192 * 2 + 1], 65),                 # one float past a chunk of the norms
    ([40 + l for l in range(32)], 32), ([40 + l for l in range(32)], 33),   # the most whose factors stage 3 works out itself
    ([33 * (l + 1) for l in range(33)], 4),               # more norms than a thread walks alone
])
def test_rows_of_any_length(sizes, Bn, give_norms):
    _check("global", _spread(Bn, sizes, Bn), 0.3, give_norms=give_norms)


def test_a_tensor_with_more_partials_than_a_warp_folds():
    sizes = [8192 * 512 + 3, 8192 * 512, 5]
    groups = _spread(3, sizes, 3)
    _check("global", groups, 0.3)
    _check("per_layer", groups, 0.2)


def test_more_tensors_than_the_largest_table():
    sizes = [40 + l % 7 for l in range(515)]
    groups = _spread(4, sizes, 9)
    _check("global", groups, 0.2)
    _check("per_layer", groups, 0.02)
