"""Calls in a second CUDA context of the same process, as a second GPU would be one: what a first context was told about the
kernels does not hold there.  In a process of its own, whose contexts end with it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import sys
import numpy as np
from cuda.bindings import driver as cu
from paper_2109_12191_b200 import binding as b

def ok(result):
    assert int(result[0]) == 0, result[0]
    return result[1] if len(result) == 2 else result[1:]

ok(cu.cuInit(0))
device = ok(cu.cuDeviceGet(0))
buffers = []

def to_gpu(array):
    address = ok(cu.cuMemAlloc(array.nbytes))
    ok(cu.cuMemcpyHtoD(address, array.ctypes.data, array.nbytes))
    buffers.append(address)
    return int(address)

def to_host(address, shape):
    out = np.empty(shape, np.float32)
    ok(cu.cuMemcpyDtoH(out.ctypes.data, address, out.nbytes))
    return out

def clip(static):
    Bn, P = 40, 5000
    G = np.random.default_rng(1).standard_normal((Bn, P), dtype=np.float32)
    n = b.dp_clip_workspace_bytes(Bn, [P])
    acc, ws = to_gpu(np.zeros(P, np.float32)), to_gpu(np.zeros(n, np.uint8))
    if static:
        b.check(b.dp_clip_accumulate_static(b.DP_CLIP_GLOBAL, Bn, [to_gpu(G)], [P], None, 50.0, [acc], None, None, stream=0))
    else:
        b.check(b.dp_clip_accumulate(b.DP_CLIP_GLOBAL, Bn, [to_gpu(G)], [P], None, 50.0, [acc], None, None, ws, n, stream=0))
    ok(cu.cuCtxSynchronize())
    d = G.astype(np.float64)
    ref = (np.minimum(1.0, 50.0 / np.linalg.norm(d, axis=1))[:, None] * d).sum(0)
    assert np.linalg.norm(to_host(acc, P) - ref) <= 2e-5 * np.linalg.norm(ref)

LAYERS = {                                                   # C_in, K_out, size, R, stride, pad
    "stem": (3, 64, 40, 3, 1, 1), "one_tile": (64, 64, 9, 1, 1, 0), "clusters": (128, 256, 9, 3, 2, 1), "gram": (256, 320, 7, 3, 1, 1),
    "shared_pixels": (64, 64, 50, 1, 1, 0),
}
kept = []

class Memory:                                                # what a batch asks of its workspace
    def __init__(self, nbytes):
        self.nbytes, self.address = nbytes, to_gpu(np.zeros(nbytes, np.uint8))
    def is_contiguous(self):
        return True
    def data_ptr(self):
        return self.address

def layer(name, dtype, seed):
    Cin, K, H, R, stride, pad = LAYERS[name]
    Bn, OH = 3, (H + 2 * pad - R) // stride + 1
    rng = np.random.default_rng(seed)
    X, dY = (rng.standard_normal(n, dtype=np.float32) for n in (Bn * H * H * Cin, Bn * OH * OH * K))
    if dtype == b.DP_BF16:
        X, dY = ((t.view(np.uint32) >> 16).astype(np.uint16) for t in (X, dY))
    return b.make_desc(b.DP_LAYER_CONV2D, dtype, Bn, Cin, K, H, H, R, R, stride, pad), to_gpu(X), to_gpu(dY), Bn, K * R * R * Cin

def conv(name, dtype, epi):
    d, X, dY, Bn, P = layer(name, dtype, 2)
    G, sq, acc = to_gpu(np.zeros((Bn, P), np.float32)), to_gpu(np.zeros(Bn, np.float32)), to_gpu(np.zeros(P, np.float32))
    n = b.dp_workspace_bytes(d, epi)
    ws = to_gpu(np.zeros(n, np.uint8))
    b.check(b.dp_per_example_wgrad(d, X, dY, G, None, sq, 1, epi, 1.0, acc, None, None, ws, n, stream=0))
    ok(cu.cuCtxSynchronize())
    return np.concatenate([to_host(t, k).ravel() for t, k in ((G, Bn * P), (sq, Bn), (acc, P))])

def batch():
    parts = [layer(name, b.DP_BF16, 3) for name in LAYERS]
    made = b.Batch([p[0] for p in parts], [b.DP_EPI_CLIP_ACCUM] * len(parts))
    kept.append(made)                                        # its streams stay with their context
    out = [(to_gpu(np.zeros(P, np.float32)), to_gpu(np.zeros(Bn, np.float32)), P, Bn) for _, _, _, Bn, P in parts]
    for i, (acc, sq, _, _) in enumerate(out):
        made.set(i, acc_w=acc, sqnorm=sq, sqnorm_stride=1)
    b.check(made.run([(X, dY) for _, X, dY, _, _ in parts], 1.0, Memory(made.workspace_bytes), stream=0))
    ok(cu.cuCtxSynchronize())
    return np.concatenate([to_host(a, n) for acc, sq, P, Bn in out for a, n in ((acc, P), (sq, Bn))])

def convs(dtype):
    return np.concatenate([conv(name, dtype, epi) for name in LAYERS for epi in range(3)])

CALLS = {"convs_bf16": lambda: convs(b.DP_BF16), "convs_f32": lambda: convs(b.DP_F32), "convs_tf32": lambda: convs(b.DP_TF32), "batch": batch,
         "clip": lambda: clip(False), "clip_static": lambda: clip(True)}
first = ok(cu.cuDevicePrimaryCtxRetain(device))
ok(cu.cuCtxSetCurrent(first))
before = CALLS[sys.argv[1]]()
second = ok(cu.cuCtxCreate(0, device))                       # current from here on
after = CALLS[sys.argv[1]]()
assert before is None or (np.array_equal(before, after) and np.all(np.isfinite(after)) and np.any(after))
print("done")
"""


def run(call):
    pytest.importorskip("cuda.bindings.driver")
    done = subprocess.run([sys.executable, "-c", PROGRAM, call], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert done.returncode == 0 and done.stdout.strip().endswith("done"), done.stdout + done.stderr


@pytest.mark.parametrize("call", ["clip", "clip_static"])
def test_flat_gradients(call):
    run(call)


@pytest.mark.parametrize("call", ["convs_bf16", "convs_f32", "convs_tf32", "batch"])
def test_weight_gradients(call):
    run(call)
