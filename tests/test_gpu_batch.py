"""A batch of layer calls of every kind against the NumPy oracle: layers of one kind share launches, blocks and scratch."""
import numpy as np
import pytest
import torch

import oracle
from paper_2109_12191_b200 import synth
from gpu_util import B, TOL_ACC_F32, TOL_FMA, TOL_NORM, dev_inputs, make_desc, oracle_layer, rel_l2, scaled_inputs

pytestmark = pytest.mark.gpu

STORE, NORM, CLIP = 0, 1, 2
LAYERS = [
    synth.conv(3, 64, 7, 2, 3, 21, False, "strided stem"), synth.conv(3, 32, 3, 1, 1, 12, True, "stem"),
    synth.conv(64, 64, 1, 1, 0, 9, False, "one tile"), synth.conv(64, 256, 3, 1, 1, 6, False, "rows of input columns"),
    synth.conv(128, 384, 1, 1, 0, 7, False, "three tiles"), synth.conv(128, 256, 3, 2, 1, 9, False, "larger clusters"),
    synth.conv(256, 320, 3, 1, 1, 7, False, "Gram matrices, one product"), synth.conv(256, 256, 3, 1, 1, 13, False, "Gram matrices, tiles"),
    synth.conv(64, 64, 3, 2, 1, 8, True, "with a bias"), synth.conv(5, 7, 3, 1, 0, 9, True, "nothing aligned"),
    synth.dense(65, 10, True, "dense"), synth.norm(24, 7), synth.norm(2048, 3), synth.norm(5, 6),
]


@pytest.mark.parametrize("Bn", [1, 5])
@pytest.mark.parametrize("dtype", ["bf16", "f32", "tf32"])
@pytest.mark.parametrize("epi,separate", [(STORE, 1), (NORM, 0), (NORM, 1), (CLIP, 0), (CLIP, 1)])
def test_layers_of_every_kind(epi, separate, dtype, Bn):
    b = B()
    inputs = [scaled_inputs(l, Bn, dtype if dtype != "tf32" else "f32", 971, i, spread=True) for i, l in enumerate(LAYERS)]
    data = [dev_inputs(inp, dtype) for inp in inputs]
    descs = [make_desc(l, Bn, dtype, 0, separate) for l in LAYERS]
    groups = [b.dp_layer_groups(d) for d in descs]
    refs = [oracle_layer(l, inp) for l, inp in zip(LAYERS, inputs)]
    sqs = []
    for (dW, db), g in zip(refs, groups):
        w, v = oracle.sqnorm(dW), (oracle.sqnorm(db) if db is not None else np.zeros(Bn))
        sqs.append(np.stack([w, v], 1) if g == 2 else (w + v)[:, None])
    C_l = float(np.sqrt(np.median(np.concatenate([s.ravel() for s in sqs]))))
    batch = b.Batch(descs, [epi] * len(LAYERS))
    out = []
    for i, (l, g) in enumerate(zip(LAYERS, groups)):
        nan = lambda *shape: torch.full(shape, float("nan"), device="cuda")  # noqa: E731
        o = dict(sqnorm=nan(Bn, g))
        if epi == STORE:
            o["G_w"], o["G_b"] = nan(Bn, l.n_weight), nan(Bn, l.n_bias) if l.n_bias else None
        if epi == CLIP:
            o["acc_w"], o["clip_out"] = torch.ones(l.n_weight, device="cuda"), nan(Bn, g)
            o["acc_b"] = torch.ones(l.n_bias, device="cuda") if l.n_bias else None
        batch.set(i, sqnorm_stride=g, **o)
        out.append(o)
    ws = torch.full((batch.workspace_bytes + 256,), 0xAB, dtype=torch.uint8, device="cuda")
    b.check(b.dp_workspace_init(ws, batch.workspace_bytes), "dp_workspace_init")
    try:
        for target in (0, 40):                               # tickets and scratch are left ready for the next run; plans stay
            b.check(b.dp_set_sm_target(target), "dp_set_sm_target")
            b.check(batch.run(data, C_l, ws[:batch.workspace_bytes]), "dp_batch_run")
    finally:
        b.dp_set_sm_target(0)
    b.check(b.dp_wgrad_check(ws), "dp_wgrad_check")
    assert bool((ws[batch.workspace_bytes:] == 0xAB).all())
    for l, d, (dW, db), sq, g, o in zip(LAYERS, descs, refs, sqs, groups, out):
        tol = TOL_ACC_F32 if dtype == "tf32" and b.dp_wgrad_uses_tensor_cores(d, epi) else TOL_FMA
        np.testing.assert_allclose(o["sqnorm"].cpu().numpy(), sq, rtol=TOL_NORM if tol == TOL_FMA else 1e-3, err_msg=l.name)
        if epi == STORE:
            assert rel_l2(o["G_w"].cpu().numpy(), dW) <= tol, l.name
            assert db is None or rel_l2(o["G_b"].cpu().numpy(), db) <= tol, l.name
        if epi == CLIP:
            f = oracle.clip_factor(sq, C_l).reshape(Bn, g)
            np.testing.assert_allclose(o["clip_out"].cpu().numpy(), f, rtol=TOL_NORM if tol == TOL_FMA else 1e-3, err_msg=l.name)
            assert rel_l2(o["acc_w"].cpu().numpy(), 1 + 2 * np.einsum("n,np->p", f[:, 0], dW)) <= tol, l.name
            assert db is None or rel_l2(o["acc_b"].cpu().numpy(), 1 + 2 * np.einsum("n,np->p", f[:, g - 1], db)) <= tol, l.name


def test_a_batch_is_planned_for_the_whole_gpu():
    """Under an SM target too, and also what it runs as calls of their own, here fused clips of biased convolutions: no
    neighbour fills what they would leave.  Same plan, same bits."""
    b, Bn, layer = B(), 24, synth.conv(64, 128, 3, 1, 1, 14, True)
    inp = scaled_inputs(layer, Bn, "bf16", 972, 0)
    d, data = make_desc(layer, Bn, "bf16"), dev_inputs(inp, "bf16")
    single, total, out = {}, {}, {}
    try:
        for target in (0, 20):
            b.check(b.dp_set_sm_target(target))
            single[target] = b.dp_workspace_bytes(d, CLIP)
            batch = b.Batch([d, d], [CLIP] * 2)
            total[target] = batch.workspace_bytes
            acc = [torch.zeros(n, device="cuda") for n in (layer.n_weight, layer.n_bias) * 2]
            sq = torch.zeros((Bn, 2), device="cuda")
            for i in range(2):
                batch.set(i, sqnorm=sq.data_ptr() + 4 * i, sqnorm_stride=2, acc_w=acc[2 * i], acc_b=acc[2 * i + 1])
            ws = torch.empty(batch.workspace_bytes, dtype=torch.uint8, device="cuda")
            b.check(b.dp_workspace_init(ws))
            b.check(batch.run([data, data], 1.0, ws))
            b.check(b.dp_wgrad_check(ws))
            out[target] = torch.cat(acc + [sq.flatten()])
    finally:
        b.dp_set_sm_target(0)
    assert single[0] != single[20]                          # a single call is planned for the target
    assert total[0] == total[20] and torch.equal(out[0], out[20])


@pytest.mark.parametrize("target", [0, 40])
@pytest.mark.parametrize("epi", [STORE, CLIP])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_calls_of_their_own_spread_over_lanes(dtype, epi, target):
    """Layers without a shared launch run side by side over the lanes, as calls of a workspace each under the SM target of the
    batch's creation: the bits are those of the single calls, from plain runs and from a replayed graph."""
    b, Bn = B(), 6
    data = [dev_inputs(scaled_inputs(l, Bn, dtype, 973, i), dtype) for i, l in enumerate(LAYERS)]
    descs = [make_desc(l, Bn, dtype, 0, 1) for l in LAYERS]
    plain, batch = b.Batch(descs, [epi] * len(LAYERS)), None
    C_l = 2.0

    def buffers(l, d):
        g = b.dp_layer_groups(d)
        o = dict(sqnorm=torch.zeros(Bn, g, device="cuda"), sqnorm_stride=g)
        if epi == STORE:
            o.update(G_w=torch.zeros(Bn, l.n_weight, device="cuda"), G_b=torch.zeros(Bn, l.n_bias, device="cuda") if l.n_bias else None)
        else:
            o.update(acc_w=torch.zeros(l.n_weight, device="cuda"), acc_b=torch.zeros(l.n_bias, device="cuda") if l.n_bias else None,
                     clip_out=torch.zeros(Bn, g, device="cuda"))
        return o

    def workspace(n):
        ws = torch.full((n + 256,), 0xAB, dtype=torch.uint8, device="cuda")
        b.check(b.dp_workspace_init(ws, n))
        return ws

    def tensors(o):
        return [t for t in o.values() if torch.is_tensor(t)]

    single, whole, laned = ([buffers(l, d) for l, d in zip(LAYERS, descs)] for _ in range(3))
    try:
        b.check(b.dp_set_sm_target(target))
        batch = b.Batch(descs, [epi] * len(LAYERS), lanes=3)
        assert batch.lanes == 3 and plain.lanes == 1
        for d, (X, dY), o in zip(descs, data, single):
            ws = workspace(b.dp_workspace_bytes(d, epi))
            b.check(b.dp_per_example_wgrad(d, X, dY, o.get("G_w"), o.get("G_b"), o["sqnorm"], o["sqnorm_stride"], epi, C_l, o.get("acc_w"),
                                           o.get("acc_b"), o.get("clip_out"), ws, ws.numel() - 256))
    finally:
        b.dp_set_sm_target(0)
    ws = [workspace(batch.workspace_bytes)] + [workspace(batch.lane_bytes) for _ in range(2)]
    views = [w[:-256] for w in ws]
    for i in range(len(LAYERS)):
        plain.set(i, **whole[i])
        batch.set(i, **laned[i])
    b.check(plain.run(data, C_l, workspace(plain.workspace_bytes)[:-256]))
    streams = [torch.cuda.Stream() for _ in range(2)]
    batch.use_lanes(streams, views[1:])
    b.check(batch.run(data, C_l, views[0]))
    torch.cuda.synchronize()
    # which layers are calls of their own: what the tensor cores do not take, and biased or fp32 fused clips
    own = [i for i, (l, d) in enumerate(zip(LAYERS, descs))
           if (l.kind == "norm" and l.Cin % 8) or l.kind == "dense" or (l.kind == "conv" and (not b.dp_wgrad_uses_tensor_cores(d, epi)
               or (epi == CLIP and (l.bias or dtype == "f32"))))]
    assert len(own) >= 3
    for i, l in enumerate(LAYERS):
        for got, want in zip(tensors(laned[i]), tensors(single[i] if i in own else whole[i])):
            assert torch.equal(got, want), l.name
    if epi == CLIP:
        for o in laned:
            o["acc_w"].zero_()
            if o["acc_b"] is not None:
                o["acc_b"].zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        b.check(batch.run(data, C_l, views[0]))
    graph.replay()
    torch.cuda.synchronize()
    for i, l in enumerate(LAYERS):
        for got, want in zip(tensors(laned[i]), tensors(single[i] if i in own else whole[i])):
            assert torch.equal(got, want), l.name
    for w in ws:
        b.check(b.dp_wgrad_check(w))
        assert bool((w[-256:] == 0xAB).all())
    batch.use_lanes(streams[:0], [])                          # no streams given: all on one, the same bits
    if epi == STORE:
        b.check(batch.run(data, C_l, views[0]))
        assert all(torch.equal(g, w) for i in own for g, w in zip(tensors(laned[i]), tensors(single[i])))


@pytest.mark.parametrize("kind", ["layered", "global"])
def test_only_the_first_lane_holds_the_batchs_scratch(kind):
    """The other lanes run one call at a time: their workspaces are those of the largest single call."""
    from paper_2109_12191_b200.step import GlobalClipStep, PerLayerClipStep
    b, layers, Bn = B(), synth.resnet_gn_layers([1, 1, 1, 1]), 2
    st = (PerLayerClipStep if kind == "layered" else GlobalClipStep)(layers, Bn, "bf16", 1.0, 1.0, lanes=4)
    epis = [CLIP] if kind == "layered" else [STORE, NORM, CLIP]
    call = max(b.dp_workspace_bytes(d, e) for d in st.descs for e in epis)
    assert [w.numel() for w in st.ws_lane] == [max(call, st.batch.workspace_bytes)] + [call] * 3
    assert call < st.batch.workspace_bytes
    largest = max(range(len(layers)), key=lambda i: b.dp_workspace_bytes(st.descs[i], epis[0]))
    X, dY = dev_inputs(synth.layer_inputs(layers[largest], Bn, "bf16", 974, 0), "bf16")
    st.begin()
    st.wgrad(largest, X, dY, lane=3)
    torch.cuda.synchronize()
    st.check()


@pytest.mark.parametrize("dtype,sizes,Bn", [
    # one pixel, one vector of channels; several channel blocks, the last one ragged; fewer pixels than a ring's stages hold
    ("bf16", [(8, 1), (24, 7), (1032, 5), (2048, 3), (512, 9), (64, 20), (2056, 2)], 3),
    ("f32", [(4, 1), (36, 6), (516, 5), (256, 4), (1024, 3)], 3),
    ("bf16", [(64, 64)], 40),                                # more items than two for every block
])
def test_normalisation_layers_beside_convolutions(dtype, sizes, Bn):
    """The form for many bytes of them: a last, large layer brings the batch there, and leaves the others in front of it."""
    b = B()
    large = synth.norm(64, 64 if Bn > 3 else 512 if dtype == "f32" else 720)
    layers = [synth.conv(256, 256, 3, 1, 1, 14)] * 4 + [synth.norm(C, H) for C, H in sizes] + [large] * (7 if Bn > 3 else 1)
    distinct = {}
    for i, l in enumerate(layers):
        if l not in distinct and l is not large:
            inp = scaled_inputs(l, Bn, dtype, 975, i, spread=True)
            distinct[l] = (inp, dev_inputs(inp, dtype))
    if large not in distinct:
        zeros = torch.zeros(large.x_shape(Bn), device="cuda", dtype=torch.bfloat16 if dtype == "bf16" else torch.float32)
        distinct[large] = (None, (zeros, zeros))
    data = [distinct[l][1] for l in layers]
    batch = b.Batch([make_desc(l, Bn, dtype, 0, 1) for l in layers], [NORM] * len(layers))
    sq = [torch.zeros((Bn, 2), device="cuda") for _ in layers]
    for i, s in enumerate(sq):
        batch.set(i, sqnorm=s, sqnorm_stride=2 if layers[i].kind == "norm" else 1)
    ws = torch.full((batch.workspace_bytes,), 0xAB, dtype=torch.uint8, device="cuda")
    b.check(b.dp_workspace_init(ws))
    for _ in range(2):                                       # items are handed out anew
        for s in sq:
            s.fill_(float("nan"))
        b.check(batch.run(data, 1.0, ws))
        for l, s in zip(layers, sq):
            inp = distinct[l][0]
            if l.kind == "norm" and inp is not None:
                dW, db = oracle_layer(l, inp)
                np.testing.assert_allclose(s.cpu().numpy(), np.stack([oracle.sqnorm(dW), oracle.sqnorm(db)], 1), rtol=TOL_NORM, err_msg=str(l))
            elif l.kind == "norm":
                assert not bool(s.any())
    b.check(b.dp_wgrad_check(ws))
