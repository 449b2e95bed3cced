"""Calls in a second CUDA context of the same process, as a second GPU would be one: what a first context was told about the
kernels does not hold there.  In a process of its own, whose contexts end with it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
import ctypes, sys
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

CALLS = {"clip": lambda: clip(False), "clip_static": lambda: clip(True)}
first = ok(cu.cuDevicePrimaryCtxRetain(device))
ok(cu.cuCtxSetCurrent(first))
CALLS[sys.argv[1]]()
second = ok(cu.cuCtxCreate(0, device))                       # current from here on
buffers.clear()
CALLS[sys.argv[1]]()
print("done")
"""


def run(call):
    pytest.importorskip("cuda.bindings.driver")
    done = subprocess.run([sys.executable, "-c", PROGRAM, call], cwd=ROOT, capture_output=True, text=True, timeout=120)
    assert done.returncode == 0 and done.stdout.strip().endswith("done"), done.stdout + done.stderr


@pytest.mark.parametrize("call", ["clip", "clip_static"])
def test_flat_gradients(call):
    run(call)
