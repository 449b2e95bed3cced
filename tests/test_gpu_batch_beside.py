"""Normalisation layers that run beside a batch's convolutions: when their blocks start, and their sums under every epilogue."""
import numpy as np
import pytest
import torch

import oracle
from paper_2109_12191_b200 import synth
from gpu_util import B, TOL_FMA, TOL_NORM, dev_inputs, kernels_of, make_desc, oracle_layer, rel_l2, scaled_inputs

pytestmark = pytest.mark.gpu

STORE, NORM, CLIP = 0, 1, 2
LARGE = synth.norm(64, 720)                                  # brings a batch of three examples to the form for many bytes


def _zeros(layer, Bn, dtype="bf16"):
    return tuple(torch.zeros(shape, device="cuda", dtype=torch.bfloat16 if dtype == "bf16" else torch.float32)
                 for shape in (layer.x_shape(Bn), layer.dy_shape(Bn)))


@pytest.mark.parametrize("lanes", [1, 2])
@pytest.mark.parametrize("convs", [
    [synth.conv(256, 320, 3, 1, 1, 7)],                      # Gram matrices and one product: nothing on the caller's stream itself
    [synth.conv(3, 64, 7, 2, 3, 21), synth.conv(64, 256, 3, 1, 1, 6), synth.conv(128, 256, 3, 2, 1, 9)],   # a regrouped input, clusters of several sizes
], ids=["gram", "mixed"])
def test_blocks_beside_convolutions_start_before_everything_else(convs, lanes):
    """Captured, the batch has one node that depends on nothing, the launch of those blocks: what started with them took their
    places on some SMs.  A copy right behind the batch can be captured too, and a replay gives the bits of the plain run."""
    runtime = pytest.importorskip("cuda.bindings.runtime")
    b, Bn = B(), 3
    layers = convs + [synth.norm(64, 20), synth.dense(65, 10, True), synth.dense(33, 7, False), LARGE]
    data = [_zeros(l, Bn) if l is LARGE else dev_inputs(scaled_inputs(l, Bn, "bf16", 976, i), "bf16") for i, l in enumerate(layers)]
    batch = b.Batch([make_desc(l, Bn, "bf16") for l in layers], [CLIP] * len(layers), lanes=lanes)
    assert batch.lanes == lanes
    sizes = [n for l in layers for n in (l.n_weight, l.n_bias)]
    ends = torch.tensor([0] + [(n + 3) // 4 * 4 for n in sizes]).cumsum(0).tolist()       # every tensor on a 16-byte boundary
    acc, sq = torch.zeros(ends[-1], device="cuda"), torch.zeros((len(layers), Bn), device="cuda")
    parts = [acc[o:o + n] for o, n in zip(ends, sizes)]
    for i in range(len(layers)):
        batch.set(i, sqnorm=sq[i], sqnorm_stride=1, acc_w=parts[2 * i], acc_b=parts[2 * i + 1] if parts[2 * i + 1].numel() else None)
    ws = torch.empty(batch.workspace_bytes, dtype=torch.uint8, device="cuda")
    b.check(b.dp_workspace_init(ws))
    if lanes > 1:
        own = torch.empty(batch.lane_bytes, dtype=torch.uint8, device="cuda")
        b.check(b.dp_workspace_init(own))
        batch.use_lanes([torch.cuda.Stream()], [own])
    copy = torch.empty_like(acc)

    b.check(batch.run(data, 1.0, ws))
    plain, plain_sq = acc.clone(), sq.clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        b.check(batch.run(data, 1.0, ws))
        copy.copy_(acc)
    err, _, roots = runtime.cudaGraphGetRootNodes(graph.raw_cuda_graph())
    assert int(err) == 0 and roots == 1
    acc.zero_()
    sq.zero_()
    graph.instantiate()
    graph.replay()
    torch.cuda.synchronize()
    b.check(b.dp_wgrad_check(ws))
    assert torch.equal(copy, plain) and torch.equal(sq, plain_sq)


def test_convolutions_with_nothing_beside_keep_their_registers():
    """Their kernels need not leave any of an SM's registers to others, and put nothing in local memory."""
    driver = pytest.importorskip("cuda.bindings.driver")
    b, Bn = B(), 3
    layers = [synth.conv(64, 64, 1, 1, 0, 9), synth.conv(64, 256, 3, 1, 1, 6), synth.conv(128, 384, 1, 1, 0, 7), synth.conv(128, 256, 3, 2, 1, 9)]
    data = [dev_inputs(scaled_inputs(l, Bn, "bf16", 977, i), "bf16") for i, l in enumerate(layers)]
    batch = b.Batch([make_desc(l, Bn, "bf16") for l in layers], [CLIP] * len(layers))
    acc, sq = [torch.zeros(l.n_weight, device="cuda") for l in layers], torch.zeros((len(layers), Bn), device="cuda")
    for i, a in enumerate(acc):
        batch.set(i, sqnorm=sq[i], sqnorm_stride=1, acc_w=a)
    ws = torch.empty(batch.workspace_bytes, dtype=torch.uint8, device="cuda")
    b.check(b.dp_workspace_init(ws))
    b.check(batch.run(data, 1.0, ws))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        b.check(batch.run(data, 1.0, ws))
    raw = driver.CUgraph(graph.raw_cuda_graph())
    err, _, count = driver.cuGraphGetNodes(raw)
    err, nodes, count = driver.cuGraphGetNodes(raw, count)
    assert int(err) == 0 and count >= 3
    for node in nodes:
        err, kind = driver.cuGraphNodeGetType(node)
        if kind != driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        err, params = driver.cuGraphKernelNodeGetParams(node)
        assert int(err) == 0
        func = params.func
        if not int(func):
            err, func = driver.cuKernelGetFunction(params.kern)
            assert int(err) == 0
        err, local = driver.cuFuncGetAttribute(driver.CUfunction_attribute.CU_FUNC_ATTRIBUTE_LOCAL_SIZE_BYTES, func)
        assert int(err) == 0 and local == 0


def test_normalisation_layers_of_small_batches_fill_gaps():
    """With few bytes of them nothing runs beside the convolutions, and no launch of the batch comes before the others."""
    driver = pytest.importorskip("cuda.bindings.driver")
    b, Bn = B(), 3
    layers = [synth.conv(64, 64, 1, 1, 0, 9), synth.conv(256, 320, 3, 1, 1, 7), synth.conv(128, 256, 3, 2, 1, 9), synth.norm(64, 20)]
    data = [dev_inputs(scaled_inputs(l, Bn, "bf16", 978, i), "bf16") for i, l in enumerate(layers)]
    batch = b.Batch([make_desc(l, Bn, "bf16") for l in layers], [CLIP] * len(layers))
    acc, sq = [torch.zeros((2, max(l.n_weight, 4)), device="cuda") for l in layers], torch.zeros((len(layers), Bn), device="cuda")
    for i, l in enumerate(layers):
        batch.set(i, sqnorm=sq[i], sqnorm_stride=1, acc_w=acc[i][0], acc_b=acc[i][1] if l.n_bias else None)
    ws = torch.empty(batch.workspace_bytes, dtype=torch.uint8, device="cuda")
    b.check(b.dp_workspace_init(ws))
    b.check(batch.run(data, 1.0, ws))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        b.check(batch.run(data, 1.0, ws))
    raw = driver.CUgraph(graph.raw_cuda_graph())
    err, _, count = driver.cuGraphGetNodes(raw)
    err, nodes, count = driver.cuGraphGetNodes(raw, count)
    priorities = set()
    for node in nodes:
        err, kind = driver.cuGraphNodeGetType(node)
        if kind == driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            err, value = driver.cuGraphKernelNodeGetAttribute(node, driver.CUlaunchAttributeID.CU_LAUNCH_ATTRIBUTE_PRIORITY)
            assert int(err) == 0
            priorities.add(value.priority)
    assert len(priorities) == 1


@pytest.mark.parametrize("H", [64, 720], ids=["apart", "beside"])
def test_lanes_count_normalisation_layers_only_where_those_follow_lane_0(H):
    """Two single calls over two lanes.  Behind large normalisation layers lane 0 would be late, so both take the other lane, one
    after the other; where those layers have a stream of their own the calls run side by side."""
    driver = pytest.importorskip("cuda.bindings.driver")
    b, Bn = B(), 3
    layers = [synth.conv(256, 256, 3, 1, 1, 14), synth.conv(5, 60, 3, 1, 0, 24), synth.conv(5, 7, 3, 1, 0, 9)] + [synth.norm(64, H)] * (1 if H > 64 else 40)
    data = [_zeros(l, Bn) for l in layers]
    descs = [make_desc(l, Bn, "bf16") for l in layers]
    assert not any(b.dp_wgrad_uses_tensor_cores(d, NORM) for d in descs[1:3])
    batch = b.Batch(descs, [NORM] * len(descs), lanes=2)
    assert batch.lanes == 2
    sq = torch.full((len(layers), Bn), 7.0, device="cuda")
    for i in range(len(layers)):
        batch.set(i, sqnorm=sq[i], sqnorm_stride=1)
    ws = [torch.empty(n, dtype=torch.uint8, device="cuda") for n in (batch.workspace_bytes, batch.lane_bytes)]
    for w in ws:
        b.check(b.dp_workspace_init(w))
    batch.use_lanes([torch.cuda.Stream()], [ws[1]])
    b.check(batch.run(data, 1.0, ws[0]))
    torch.cuda.synchronize()
    assert not bool(sq.any())
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        b.check(batch.run(data, 1.0, ws[0]))
    raw = driver.CUgraph(graph.raw_cuda_graph())
    err, _, _, _, count = driver.cuGraphGetEdges_v2(raw)
    err, start, end, _, count = driver.cuGraphGetEdges_v2(raw, count)
    assert int(err) == 0
    before = {}
    for a, z in zip(start, end):
        before.setdefault(int(z), []).append(a)

    def name(node):
        err, kind = driver.cuGraphNodeGetType(node)
        if kind != driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            return b""
        err, params = driver.cuGraphKernelNodeGetParams(node)
        return driver.cuKernelGetName(params.kern)[1] if int(params.kern) else driver.cuFuncGetName(params.func)[1]

    def follows_one(node):
        return any(b"conv_wgrad_fma" in name(a) or follows_one(a) for a in before.get(int(node), []))

    own = {int(n): n for n in list(start) + list(end) if b"conv_wgrad_fma" in name(n)}
    assert len(own) == 2
    assert sum(follows_one(n) for n in own.values()) == (0 if H > 64 else 1)


@pytest.mark.parametrize("epi,separate", [(STORE, 1), (CLIP, 0), (CLIP, 1)])
@pytest.mark.parametrize("dtype,sizes,Bn", [
    # one pixel, one vector of channels; several channel blocks, the last one ragged; fewer pixels than a ring's stages hold
    ("bf16", [(8, 1), (24, 7), (1032, 5), (2048, 3), (512, 9), (64, 20), (2056, 2)], 3),
    ("f32", [(4, 1), (36, 6), (516, 5), (256, 4), (1024, 3)], 3),
])
def test_gradients_and_clipped_sums_of_layers_beside_convolutions(dtype, sizes, Bn, epi, separate):
    b = B()
    large = LARGE if dtype == "bf16" else synth.norm(64, 512)
    norms = [synth.norm(C, H) for C, H in sizes]
    layers = [synth.conv(256, 256, 3, 1, 1, 14)] * 4 + norms + [large]
    inputs = [scaled_inputs(l, Bn, dtype, 979, i) if l in norms else None for i, l in enumerate(layers)]
    data = [_zeros(l, Bn, dtype) if inp is None else dev_inputs(inp, dtype) for l, inp in zip(layers, inputs)]
    refs = [oracle_layer(l, inp) if inp is not None else None for l, inp in zip(layers, inputs)]
    sqs = [None if r is None else np.stack([oracle.sqnorm(r[0]), oracle.sqnorm(r[1])], 1) for r in refs]
    sqs = [s if s is None or separate else s.sum(1, keepdims=True) for s in sqs]
    C_l = float(np.sqrt(np.median(np.concatenate([s.ravel() for s in sqs if s is not None]))))
    batch = b.Batch([make_desc(l, Bn, dtype, 0, separate) for l in layers], [epi if l.kind == "norm" else NORM for l in layers])
    out = []
    for i, l in enumerate(layers):
        g = 1 + separate if l.kind == "norm" else 1
        o = dict(sqnorm=torch.full((Bn, g), float("nan"), device="cuda"))
        if l.kind == "norm" and epi == STORE:
            o.update(G_w=torch.full((Bn, l.n_weight), float("nan"), device="cuda"), G_b=torch.full((Bn, l.n_bias), float("nan"), device="cuda"))
        if l.kind == "norm" and epi == CLIP:
            o.update(acc_w=torch.ones(l.n_weight, device="cuda"), acc_b=torch.ones(l.n_bias, device="cuda"), clip_out=torch.full((Bn, g), float("nan"), device="cuda"))
        batch.set(i, sqnorm_stride=g, **o)
        out.append(o)
    ws = torch.full((batch.workspace_bytes + 256,), 0xAB, dtype=torch.uint8, device="cuda")
    b.check(b.dp_workspace_init(ws, batch.workspace_bytes))
    for _ in range(2):                                       # items are handed out anew
        b.check(batch.run(data, C_l, ws[:batch.workspace_bytes]))
    b.check(b.dp_wgrad_check(ws))
    assert any("affine_batch_stream_kernel" in name for name in kernels_of(lambda: b.check(batch.run(data, C_l, ws[:batch.workspace_bytes]))))
    assert bool((ws[batch.workspace_bytes:] == 0xAB).all())
    for l, ref, sq, o in zip(layers, refs, sqs, out):
        if ref is None:
            continue
        np.testing.assert_allclose(o["sqnorm"].cpu().numpy(), sq, rtol=TOL_NORM, err_msg=str(l))
        if epi == STORE:
            assert rel_l2(o["G_w"].cpu().numpy(), ref[0]) <= TOL_FMA and rel_l2(o["G_b"].cpu().numpy(), ref[1]) <= TOL_FMA, str(l)
        else:
            f = oracle.clip_factor(sq, C_l).reshape(Bn, -1)
            np.testing.assert_allclose(o["clip_out"].cpu().numpy(), f, rtol=TOL_NORM, err_msg=str(l))
            assert rel_l2(o["acc_w"].cpu().numpy(), 1 + 2 * np.einsum("n,np->p", f[:, 0], ref[0])) <= TOL_FMA, str(l)
            assert rel_l2(o["acc_b"].cpu().numpy(), 1 + 2 * np.einsum("n,np->p", f[:, -1], ref[1])) <= TOL_FMA, str(l)
