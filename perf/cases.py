"""Performance cases: what users of this library run, through its public entry points.

Every case is one pass of one of these uses:

  global   one step of whole-model clipping with ``GlobalClipStep`` (begin, the chunks, finish)
  layered  one step of per-layer clipping with ``PerLayerClipStep`` (begin, the chunks, finish)
  flat     one step over flattened per-example gradients with ``FlatClipStep``
  wgrad    per-example weight-gradient calls, layer after layer, with one of the three epilogues
  grouped  clipping of stored gradients, the parameter tensors gathered into groups (pipeline stages)
  update   noise, average and the SGD update of the parameters in one call

Shapes are those of the workloads in ``synth`` or generic ones of the same kind.  Per-example gradients have norms
spread over a decade around the clipping threshold, so that some examples are clipped and some are not.
"""
import math

import torch

from paper_2109_12191_b200 import binding as b
from paper_2109_12191_b200 import synth
from paper_2109_12191_b200.step import FlatClipStep, GlobalClipStep, PerLayerClipStep, layer_desc

_EPILOGUES = {"store": b.DP_EPI_STORE_NORM, "norm": b.DP_EPI_NORM_ONLY, "clip": b.DP_EPI_CLIP_ACCUM}


def listed():
    R50 = synth.RESNET50_GN_PARAMS
    return [
        # a single dense layer and a handful of examples: nothing but latency and launches
        dict(name="dense_b8", use="global", model="dense", Cin=256, Kout=64, B=8, chunks=1, dtype="f32", lanes=1,
             recompute="none", sms=0, graph=False),
        # a small image classifier at its full batch, tuned as in the benchmark: four streams, the classifier's gradients
        # recomputed, tf32 tensor cores, the static part of the step replayed from a CUDA graph
        dict(name="cnn_b256_graph", use="global", model="cnn", size=32, w1=32, w2=64, w3=128, B=256, chunks=1, dtype="tf32",
             lanes=4, recompute="auto", sms=2, graph=True),
        # the same classifier as a first program writes it: default options, fp32, a small batch, plain calls
        dict(name="cnn_b32", use="global", model="cnn", size=32, w1=32, w2=64, w3=128, B=32, chunks=1, dtype="f32",
             lanes=1, recompute="none", sms=0, graph=False),
        # ResNet-50 at 224 x 224 with per-layer clipping, tuned as in the benchmark: 16 streams and graph replay
        dict(name="r50_layered_b32_graph", use="layered", model="resnet", n1=3, n2=4, n3=6, n4=3, B=32, chunks=2, lanes=16,
             sms=1, graph=True),
        # the same with default options and a chunk that leaves room for the activations of a large model
        dict(name="r50_layered_b8", use="layered", model="resnet", n1=3, n2=4, n3=6, n4=3, B=8, chunks=1, lanes=1, sms=0,
             graph=False),
        # ResNet-50 with whole-model clipping, every layer's per-example gradients kept
        dict(name="r50_global_b16", use="global", model="resnet", n1=3, n2=4, n3=6, n4=3, B=16, chunks=1, dtype="bf16", lanes=1,
             recompute="none", sms=0, graph=False),
        # flattened ResNet-50 gradients that come from elsewhere, two accumulated chunks: memory from end to end
        dict(name="flat_r50_b64", use="flat", P=R50, B=64, chunks=2, micro=1, norms="computed", noise="once"),
        # flattened gradients of the small classifier: many short rows that start at any address
        dict(name="flat_cnn_b256", use="flat", P=175178, B=256, chunks=1, micro=1, norms="computed", noise="once"),
        # a noise draw per example, the form of the paper's own implementation
        dict(name="flat_noised_b32", use="flat", P=8000000, B=32, chunks=1, micro=1, norms="computed", noise="example"),
        # norms of eight representative ResNet-50 layers (first pass of whole-model clipping without stored gradients)
        dict(name="sweep_norm_b32", use="wgrad", model="sweep", B=32, dtype="bf16", epilogue="norm"),
        # stored ResNet-50 gradients clipped by four pipeline stages
        dict(name="grouped_r50_b16", use="grouped", model="resnet", n1=3, n2=4, n3=6, n4=3, B=16, groups=4),
        # the end of a ResNet-50 training step: noise, average, momentum update
        dict(name="update_r50", use="update", P=R50, momentum=0.9),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    use = rng.choice(["dense", "cnn", "layered", "resnet", "flat", "wgrad", "grouped", "update"])
    if use == "dense":
        B, Cin = _log(rng, 1, 256), _log(rng, 16, 4096)
        return dict(use="global", model="dense", Cin=Cin, Kout=_log(rng, 8, 1000), B=B, chunks=rng.randint(1, 2),
                    dtype=rng.choice(["f32", "bf16"]), lanes=1, recompute=rng.choice(["none", "auto"]), sms=0, graph=False)
    if use == "cnn":
        tuned = rng.random() < 0.5
        return dict(use="global", model="cnn", size=rng.randint(24, 48), w1=rng.choice([32, 64]), w2=rng.choice([64, 128]),
                    w3=rng.choice([128, 192, 256]), B=_log(rng, 8, 256), chunks=1, dtype=rng.choice(["f32", "tf32"]),
                    lanes=4 if tuned else 1, recompute="auto" if tuned else "none", sms=2 if tuned else 0, graph=tuned)
    blocks = dict(n1=rng.randint(1, 3), n2=rng.randint(1, 4), n3=rng.randint(1, 9), n4=rng.randint(1, 3))
    if use == "layered":
        tuned = rng.random() < 0.5
        return dict(use="layered", model="resnet", **blocks, B=_log(rng, 2, 32), chunks=rng.randint(1, 2),
                    lanes=16 if tuned else 1, sms=1 if tuned else 0, graph=tuned)
    if use == "resnet":
        return dict(use="global", model="resnet", **blocks, B=_log(rng, 2, 16), chunks=1, dtype="bf16", lanes=1,
                    recompute="none", sms=0, graph=False)
    if use == "flat":
        form = rng.choice(["computed", "computed", "supplied", "micro", "noised"])
        P = _log(rng, 10000, 25600000)
        most = min(256, (250000000 if form == "noised" else 1600000000) // P)
        B = _log(rng, 2, most)
        return dict(use="flat", P=P, B=B - B % 2 if form == "micro" else B, chunks=1 if form == "noised" else rng.randint(1, 2),
                    micro=2 if form == "micro" else 1, norms="supplied" if form == "supplied" else "computed",
                    noise="example" if form == "noised" else "once")
    if use == "wgrad":
        R = rng.choice([1, 3])
        return dict(use="wgrad", model="conv", Cin=64 * _log(rng, 1, 8), Kout=64 * _log(rng, 1, 8), R=R,
                    stride=rng.choice([1, 1, 2]), size=_log(rng, 7, 56), B=_log(rng, 2, 32), dtype="bf16",
                    epilogue=rng.choice(sorted(_EPILOGUES)))
    if use == "grouped":
        return dict(use="grouped", model="resnet", **blocks, B=_log(rng, 2, 16), groups=rng.randint(1, 8))
    return dict(use="update", P=_log(rng, 10000, 100000000), momentum=rng.choice([0.0, 0.9]))


def _layers(case):
    if case["model"] == "dense":
        return [synth.dense(case["Cin"], case["Kout"], True)]
    if case["model"] == "cnn":
        w1, w2, w3, size = case["w1"], case["w2"], case["w3"], case["size"]
        c2 = synth.conv(w1, w2, 3, 2, 1, size, True)
        c3 = synth.conv(w2, w3, 3, 2, 1, c2.OH, True)
        return [synth.conv(3, w1, 3, 1, 1, size, True), c2, c3, synth.dense(w3 * c3.OH * c3.OW, 10, True)]
    if case["model"] == "resnet":
        return synth.resnet_gn_layers([case["n1"], case["n2"], case["n3"], case["n4"]])
    if case["model"] == "sweep":
        return synth.resnet50_sweep()["layers"]
    return [synth.conv(case["Cin"], case["Kout"], case["R"], case["stride"], case["R"] // 2, case["size"])]


def _inputs(layers, B, dtype, gen, C, per_layer):
    """(X, dY) of every layer, N(0,1) up to one factor per example that spreads the gradients' norms around the threshold."""
    kind = torch.bfloat16 if dtype == "bf16" else torch.float32
    spread = torch.pow(10.0, torch.rand(B, device="cuda", generator=gen) - 0.5)
    whole = math.sqrt(sum(l.flops() / 2 for l in layers))
    out = []
    for l in layers:
        X = torch.empty(l.x_shape(B), device="cuda", dtype=kind).normal_(generator=gen)
        dY = torch.empty(l.dy_shape(B), device="cuda", dtype=kind).normal_(generator=gen)
        norm = math.sqrt(l.flops() / 2) if per_layer else whole
        dY *= (spread * (C / norm)).to(kind).reshape((B,) + (1,) * (dY.dim() - 1))
        out.append((X, dY))
    return out


def _gradients(sizes, B, gen, C):
    """Per-example gradients of the given tensor sizes, whole-gradient norms spread around C."""
    spread = torch.pow(10.0, torch.rand((B, 1), device="cuda", generator=gen) - 0.5) * (C / math.sqrt(sum(sizes)))
    out = []
    for p in sizes:
        G = torch.empty((B, p), device="cuda").normal_(generator=gen)
        out.append(G.mul_(spread))
    return out


def _sizes(layers):
    return [n for l in layers for n in (l.n_weight, l.n_bias) if n]


def _set_sms(fraction):
    """0: every call has the GPU to itself; k: calls run side by side, each told to take 1/k of the SMs."""
    sms = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count
    b.check(b.dp_set_sm_target(sms // fraction if fraction else 0), "dp_set_sm_target")


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    use, B = case["use"], case.get("B")
    s = dict(case=case, use=use, seed=seed, step=0)
    _set_sms(case.get("sms", 0))
    if use in ("global", "layered"):
        layers = _layers(case)
        if use == "global":
            obj = GlobalClipStep(layers, B, case["dtype"], 1.0, 1.0, lanes=case["lanes"], recompute=case["recompute"])
            s["chunks"] = [_inputs(layers, B, case["dtype"], gen, 1.0, False) for _ in range(case["chunks"])]
        else:
            obj = PerLayerClipStep(layers, B, "bf16", 1.0, 1.0, lanes=case["lanes"])
            s["chunks"] = [_inputs(layers, B, "bf16", gen, obj.C_l, True) for _ in range(case["chunks"])]
        s["obj"] = obj
        if case["graph"]:
            # the static part of the step, captured once; a first pass runs the calls before the capture
            _plain_chunks(s)
            torch.cuda.synchronize()
            s["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(s["graph"]):
                _plain_chunks(s)
    elif use == "flat":
        s["obj"] = FlatClipStep(case["P"], B, 1.0, 1.0, per_example_noise=case["noise"] == "example", micro=case["micro"])
        s["chunks"] = [_gradients([case["P"]], B, gen, 1.0)[0] for _ in range(case["chunks"])]
        s["sq"] = [torch.linalg.vector_norm(G, dim=1, keepdim=True).square_() if case["norms"] == "supplied" else None
                   for G in s["chunks"]]
    elif use == "wgrad":
        layers, epi = _layers(case), _EPILOGUES[case["epilogue"]]
        s["epi"], s["calls"] = epi, []
        for l, (X, dY) in zip(layers, _inputs(layers, B, case["dtype"], gen, 1.0, True)):
            d = layer_desc(l, B, case["dtype"], bias_separate=0)
            ws = torch.empty(b.dp_workspace_bytes(d, epi), dtype=torch.uint8, device="cuda")
            b.check(b.dp_workspace_init(ws), "dp_workspace_init")
            s["calls"].append(dict(desc=d, X=X, dY=dY, ws=ws, sq=torch.zeros((B, 1), device="cuda"),
                                   G=torch.empty((B, l.n_weight), device="cuda") if case["epilogue"] == "store" else None,
                                   acc=torch.zeros(l.n_weight, device="cuda") if case["epilogue"] == "clip" else None))
    elif use == "grouped":
        sizes = _sizes(_layers(case))
        s["P_l"], s["G"] = sizes, _gradients(sizes, B, gen, 1.0)
        s["group_of"] = [min(case["groups"] - 1, i * case["groups"] // len(sizes)) for i in range(len(sizes))]
        s["acc"] = torch.zeros(sum((p + 3) // 4 * 4 for p in sizes), device="cuda")
        starts = [0]
        for p in sizes:
            starts.append(starts[-1] + (p + 3) // 4 * 4)
        s["views"] = [s["acc"][o:o + p] for o, p in zip(starts, sizes)]
        s["norms"] = torch.zeros((B, case["groups"]), device="cuda")
        s["ws"] = torch.empty(b.dp_clip_workspace_bytes(B, sizes), dtype=torch.uint8, device="cuda")
    else:
        P = case["P"]
        s["acc"] = torch.empty(P, device="cuda").normal_(0.0, 1.0, generator=gen)
        s["theta"] = torch.empty(P, device="cuda").normal_(0.0, 0.02, generator=gen)
        s["mom"] = torch.zeros(P, device="cuda") if case["momentum"] else None
    return s


def _plain_chunks(s):
    obj = s["obj"]
    obj.begin()
    for inputs in s["chunks"]:
        obj.chunk(inputs)


def run(s):
    case, use = s["case"], s["use"]
    s["step"] += 1                                  # every training step draws its own noise
    if use in ("global", "layered"):
        obj = s["obj"]
        if case["graph"]:
            s["graph"].replay()
        else:
            _plain_chunks(s)
        out = obj.finish(seed=s["seed"], step=s["step"], total_batch=case["B"] * case["chunks"])
        if use == "global":
            return {"grad": out, "sqnorms": obj.sq, "norms": obj.norms, "factors": obj.clip}
        # per-layer clipping averages in place: all tensors' results lie in the one accumulator
        return {"grad": obj.acc, "sqnorms": obj.sq}
    if use == "flat":
        obj, total = s["obj"], case["B"] * case["chunks"]
        obj.begin(total_batch=total, seed=s["seed"], step=s["step"])
        for G, sq in zip(s["chunks"], s["sq"]):
            obj.chunk(G, sq)
        grad = obj.finish(seed=s["seed"], step=s["step"], total_batch=total)
        runs = case["B"] // case["micro"]           # one norm and factor for every clipped unit
        return {"grad": grad, "norms": obj.norms[:runs], "factors": obj.clip[:runs]}
    if use == "wgrad":
        for c in s["calls"]:
            if c["acc"] is not None:
                c["acc"].zero_()
            b.check(b.dp_per_example_wgrad(c["desc"], c["X"], c["dY"], c["G"], None, c["sq"], 1, s["epi"], 1.0, c["acc"], None,
                                           None, c["ws"]), "dp_per_example_wgrad")
        return [[c["sq"], c["G"], c["acc"]] for c in s["calls"]]
    if use == "grouped":
        s["acc"].zero_()
        b.check(b.dp_clip_accumulate_grouped(case["B"], case["groups"], s["group_of"], s["G"], s["P_l"], None, 1.0, s["views"],
                                             s["norms"], None, s["ws"]), "dp_clip_accumulate_grouped")
        return {"acc": s["acc"], "norms": s["norms"]}
    b.check(b.dp_noise_average_sgd(s["acc"], case["P"], 0, 1.0, 1.0, 1024, s["seed"], s["step"], 0.1, case["momentum"], s["theta"],
                                   s["mom"]), "dp_noise_average_sgd")
    return {"theta": s["theta"], "momentum": s["mom"]}


def work(case):
    """Each input read once, each result written once; multiply-adds counted as two."""
    use, B, chunks = case["use"], case.get("B"), case.get("chunks", 1)
    if use in ("global", "layered", "wgrad"):
        layers = _layers(case)
        size = 2 if case.get("dtype", "bf16") == "bf16" else 4
        read = sum(math.prod(l.x_shape(B)) + math.prod(l.dy_shape(B)) for l in layers) * size * chunks
        flops = sum(l.flops() for l in layers) * B * chunks
        P = sum(_sizes(layers))
        if use == "wgrad":
            written = 4 * B * len(layers) + {"store": 4 * B * P, "norm": 0, "clip": 4 * P}[case["epilogue"]]
        else:
            written = 4 * P + 4 * B * len(_sizes(layers))
        return {"bytes": read + written, "flops": flops}
    if use == "flat":
        return {"bytes": 4 * case["P"] * (B * chunks + 1), "flops": 4 * case["P"] * B * chunks}
    if use == "grouped":
        P = sum(_sizes(_layers(case)))
        return {"bytes": 4 * P * (B + 1), "flops": 4 * P * B}
    return {"bytes": 4 * case["P"] * (5 if case["momentum"] else 3), "flops": 10 * case["P"]}


def tolerance(case):
    """fp32 sums of fp32 products differ by their order only.  bf16 inputs have exact products, summed in fp32 (and the
    per-example norms of all forms agree to 1e-4).  The tf32 option rounds its inputs to eleven significant bits."""
    if case.get("dtype") == "tf32":
        return {"rel": 1e-3}
    if case["use"] == "layered" or case.get("dtype") == "bf16":
        return {"rel": 1e-4}
    return {"rel": 2e-5}
