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
