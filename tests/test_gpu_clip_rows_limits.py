"""Flat gradients read once, where waits run out and where rows, norms and thresholds leave the range of numbers."""
import pytest
import torch

from gpu_util import B as binding, TOL_FMA, TOL_NORM

pytestmark = pytest.mark.gpu


def run(b, G, C, norms=None, clip=None):
    Bn, P = G.shape
    acc = torch.ones(P, device="cuda")
    n = b.dp_clip_workspace_bytes(Bn, [P])
    ws = torch.full((n,), 0xAB, dtype=torch.uint8, device="cuda")
    b.check(b.dp_clip_accumulate(b.DP_CLIP_GLOBAL, Bn, [G], [P], None, C, [acc], norms, clip, ws))
    torch.cuda.synchronize()
    return acc


# blocks a cluster: one; one, one cluster in all; two, one cluster; four; eight, rows of every register's worth; eight, some of them empty
@pytest.mark.parametrize("Bn,P", [(300, 2048), (1, 100), (1, 12000), (700, 98304), (19, 196608), (12, 131073)])
def test_a_wait_that_gives_up_leaves_nothing_that_looks_right(Bn, P):
    b = binding()
    G = torch.randn((Bn, P), device="cuda", generator=torch.Generator(device="cuda").manual_seed(P))
    C = 0.5 * P ** 0.5
    norms, clip = torch.zeros(Bn, device="cuda"), torch.zeros(Bn, device="cuda")
    b.dp_debug_set_wait_polls(0)
    try:
        acc = run(b, G, C, norms, clip)
    finally:
        b.dp_debug_set_wait_polls(-1)
    assert bool(torch.isnan(acc).all()) and bool(torch.isnan(norms).all()) and bool(torch.isnan(clip).all())
    acc = run(b, G, C, norms, clip)
    d = G.double()
    norm = torch.linalg.vector_norm(d, dim=1)
    f = torch.clamp(C / norm, max=1.0)
    torch.testing.assert_close(norms.double(), norm, rtol=TOL_NORM, atol=0.0)
    torch.testing.assert_close(clip.double(), f, rtol=TOL_NORM, atol=0.0)
    ref = 1 + (f[:, None] * d).sum(0)
    assert float(torch.linalg.vector_norm(acc.double() - ref) / torch.linalg.vector_norm(ref)) <= TOL_FMA


@pytest.mark.parametrize("C", [float("inf"), 3e38, 1.0, 1e-30, 1e-41])
@pytest.mark.parametrize("special", [None, float("inf"), float("nan")])
@pytest.mark.parametrize("Bn,P", [(300, 2048), (19, 131071)])
def test_numbers_past_their_range_as_in_two_passes(Bn, P, special, C):
    """Rows with an infinity or a NaN at either end, rows of zeros, rows whose squared norm overflows or vanishes, and thresholds
    of any size: what the general path makes of them (one group of one tensor always goes that way)."""
    b = binding()
    G = torch.randn((Bn, P), device="cuda", generator=torch.Generator(device="cuda").manual_seed(P))
    G[1] = 0.0
    G[2] *= 1e25
    G[3] *= 1e-25
    if special is not None:
        G[4, 0] = special
        G[5, P - 1] = special
    out = [[torch.full((Bn,), -1.0, device="cuda") for _ in range(2)] for _ in range(2)]
    once = run(b, G, C, *out[0])
    twice = torch.ones(P, device="cuda")
    ws = torch.empty(b.dp_clip_workspace_bytes(Bn, [P]), dtype=torch.uint8, device="cuda")
    b.check(b.dp_clip_accumulate_grouped(Bn, 1, [0], [G], [P], None, C, [twice], *out[1], ws))
    for one, two in zip(out[0], out[1]):
        torch.testing.assert_close(one, two, rtol=TOL_NORM, atol=1e-44, equal_nan=True)
    assert bool((torch.isnan(once) == torch.isnan(twice)).all()) and bool((torch.isinf(once) == torch.isinf(twice)).all())
    finite = torch.isfinite(twice)
    error = torch.linalg.vector_norm(once[finite].double() - twice[finite].double())
    assert float(error) <= TOL_FMA * float(torch.linalg.vector_norm(twice[finite].double()))
