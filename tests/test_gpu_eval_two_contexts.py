"""The network calls' kept scratch belongs to the CUDA context that is current:
with several contexts on one device, made and destroyed between calls, a call
never touches memory of another one (or of one that is gone).  Runs in a process
of its own, on the driver API."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import ctypes as C
import numpy as np
from paper_2301_05780_gb300 import pdds, workloads as W

cu = C.CDLL("libcuda.so.1")
L = pdds.lib()
vp = C.c_void_p


def ck(r):
    assert r == 0, r


def alloc(nbytes):
    p = C.c_uint64()
    ck(cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(nbytes)))
    return p.value


def up(a):
    p = alloc(a.nbytes)
    ck(cu.cuMemcpyHtoD_v2(C.c_uint64(p), a.ctypes.data_as(vp), C.c_size_t(a.nbytes)))
    return p


def down(p, a):
    ck(cu.cuMemcpyDtoH_v2(a.ctypes.data_as(vp), C.c_uint64(p), C.c_size_t(a.nbytes)))
    return a


r = np.random.default_rng(1)
theta = W.mlp_init().astype(np.float32)
xy = r.uniform(-1, 1, (5000, 2)).astype(np.float32)
guard = r.integers(0, 255, 1 << 20).astype(np.uint8)


def evaluate():
    """v and grad v by both engines, with live buffers of the context's own around the calls."""
    live = [up(guard) for _ in range(24)]
    t, x = up(theta), up(xy)
    out = []
    for f in (L.pdds_mlp_eval_tc, L.pdds_mlp_eval):
        v, g = alloc(4 * len(xy)), alloc(8 * len(xy))
        f.argtypes = [vp, vp, C.c_int64, vp, vp, vp]
        st = f(t, x, len(xy), v, g, None)
        assert st == pdds.PDDS_OK, (st, L.pdds_last_error(None))
        out += [down(v, np.empty(len(xy), np.float32)), down(g, np.empty((len(xy), 2), np.float32))]
    got = np.empty_like(guard)
    for p in live:
        assert np.array_equal(down(p, got), guard)
    return out


ck(cu.cuInit(0))
dev = C.c_int()
ck(cu.cuDeviceGet(C.byref(dev), 0))
primary = vp()
ck(cu.cuDevicePrimaryCtxRetain(C.byref(primary), dev))
ck(cu.cuCtxSetCurrent(primary))
want = evaluate()
for turn in range(3):
    ctx = vp()
    ck(cu.cuCtxCreate_v2(C.byref(ctx), 0, dev))   # becomes current
    for a, b in zip(evaluate(), want):
        assert np.array_equal(a, b)
    ck(cu.cuCtxSetCurrent(primary))
    for a, b in zip(evaluate(), want):
        assert np.array_equal(a, b)
    ck(cu.cuCtxDestroy_v2(ctx))
print("contexts ok")
'''


def test_network_calls_in_several_contexts():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "contexts ok" in r.stdout, r.stdout + r.stderr
