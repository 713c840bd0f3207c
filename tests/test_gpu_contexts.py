"""A process may have several contexts on a device: what is set once per kernel has to be set in each of them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import ctypes as C
from cuda.bindings import driver as cu
from paper_2403_04643_b200 import qaq

def ok(r):
    assert r[0] == cu.CUresult.CUDA_SUCCESS, r
    return r[1] if len(r) > 1 else None

def calls():
    # kernels with more than 48 KB of shared memory: thresholds of a short sequence, score window, decode, compaction
    BH, T, D, W = 4, 128, 128, 32
    cfg, h = qaq.make_config(1, BH, D, 2 * T, 2, 8, W, 0.01), C.c_void_p()
    def alloc(n):
        p = ok(cu.cuMemAlloc(n))
        ok(cu.cuMemsetD8(p, 0, n))
        return int(p)
    K, V, q, out, thr, bits = alloc(BH * T * D * 2), alloc(BH * T * D * 2), alloc(BH * W * D * 2), alloc(BH * D * 4), alloc(BH * 16), alloc(BH * T)
    ring, nv, ws, n = alloc(BH * W * T * 4), alloc(BH * T), alloc(64 << 20), 64 << 20
    st = [L.qaq_cache_create(C.byref(cfg), C.byref(h)),
          L.qaq_outlier_thresholds(C.byref(cfg), K, V, BH * T * D, T * D, D, T, thr, ws, n, None),
          L.qaq_prefill_window(C.byref(cfg), q, K, BH * T * D, T * D, D, T, 0.1, ring, nv, None, ws, n, None),
          L.qaq_quantize_append(h, K, V, BH * T * D, T * D, D, T, bits, bits, None, None, None, thr, None),
          L.qaq_decode_attention(h, q, 0.1, out, None, ws, n, None),
          L.qaq_cache_compact(h, None)]
    ok(cu.cuCtxSynchronize())
    assert st == [0] * 6, (st, L.qaq_last_cuda_error())
    L.qaq_cache_destroy(h)

ok(cu.cuInit(0))
dev, L = ok(cu.cuDeviceGet(0)), qaq.lib()
first = ok(cu.cuDevicePrimaryCtxRetain(dev))
ok(cu.cuCtxSetCurrent(first))
calls()
for _ in range(2):
    try:
        other = ok(cu.cuCtxCreate(0, dev))
    except TypeError:                    # newer bindings take creation parameters first
        other = ok(cu.cuCtxCreate(None, 0, dev))
    calls()
    calls()
    ok(cu.cuCtxDestroy(other))
    ok(cu.cuCtxSetCurrent(first))
    calls()
print("ok")
"""


def test_the_same_calls_in_contexts_that_come_and_go():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split()[-1:] == ["ok"], r.stderr[-2000:]
