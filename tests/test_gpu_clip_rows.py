"""Flat gradients whose rows go through a cluster once: at the edges of chunks, clusters and rings, rows and
matrices starting at any word, against float64."""
import pytest
import torch

from gpu_util import B as binding, TOL_FMA, TOL_NORM

pytestmark = pytest.mark.gpu

CHUNK = 2048
MOST = 8 * 48 * 512


@pytest.mark.parametrize("Bn,P,lead", [
    (1, 1, 0), (3, 2, 3), (5, 7, 1), (2, CHUNK - 1, 2), (300, CHUNK, 0), (37, CHUNK + 1, 1), (150, 4 * CHUNK + 3, 3), (90, 6 * CHUNK - 1, 1),
    (1000, 8 * CHUNK - 2, 2), (9, 12 * CHUNK, 0), (620, 12 * CHUNK + 1, 2), (320, 24 * CHUNK + 6, 1), (170, 48 * CHUNK - 2, 3),
    (35, 48 * CHUNK + 1, 0), (40, 64 * CHUNK + 5, 1), (19, MOST - 1, 3), (6, MOST, 0), (4, MOST + 1, 1), (40, 40 * CHUNK, 2)])
def test_rows_read_once(Bn, P, lead):
    b = binding()
    gen = torch.Generator(device="cuda").manual_seed(1000 * Bn + P)
    # the matrix ends with its allocation or starts inside it: nothing around it may be read
    store = torch.full((lead + Bn * P + 4,), float("nan"), device="cuda")
    G = store[lead:lead + Bn * P].view(Bn, P)
    G.normal_(generator=gen)
    G *= torch.pow(10.0, torch.rand((Bn, 1), device="cuda", generator=gen) * 2 - 1)
    if Bn > 4:
        G[3] = 0.0                                           # factor 1
        G[4] *= 1e25                                         # a squared norm past fp32's range: nothing is left of it
    C = float(P) ** 0.5
    acc = torch.ones(P + 8, device="cuda")
    norms, clip = torch.full((Bn,), -1.0, device="cuda"), torch.full((Bn,), -1.0, device="cuda")
    n = b.dp_clip_workspace_bytes(Bn, [P])
    ws = torch.full((n + 256,), 0xAB, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        b.check(b.dp_clip_accumulate(b.DP_CLIP_GLOBAL, Bn, [G.data_ptr()], [P], None, C, [acc.data_ptr()], norms, clip, ws[:n], n))
    d = G.double()
    norm = torch.linalg.vector_norm(d, dim=1)
    f = torch.clamp(C / norm, max=1.0)
    if Bn > 4:
        f[4] = 0.0
        norm[4] = float("inf")
    torch.testing.assert_close(norms.double(), norm, rtol=TOL_NORM, atol=0.0)
    torch.testing.assert_close(clip.double(), f, rtol=TOL_NORM, atol=0.0)
    ref = 1 + 2 * (f[:, None] * d).sum(0)
    assert float(torch.linalg.vector_norm(acc[:P].double() - ref) / torch.linalg.vector_norm(ref)) <= TOL_FMA
    assert bool((acc[P:] == 1.0).all()) and bool((ws[n:] == 0xAB).all())
    # the general path, with a workspace that has no room for the clusters' sums: the same but for the order of sums
    general = b.dp_clip_workspace_bytes(Bn, [P, 1]) if n > 4096 else n
    again = torch.zeros(P, device="cuda")
    b.check(b.dp_clip_accumulate(b.DP_CLIP_PER_LAYER, Bn, [G.data_ptr()], [P], None, C, [again.data_ptr()], None, None, ws, min(general, n)))
    assert float(torch.linalg.vector_norm(2 * again.double() + 1 - acc[:P].double()) / torch.linalg.vector_norm(ref)) <= TOL_FMA
