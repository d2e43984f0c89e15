"""Handles in two CUDA contexts of one device, one after the other: a
destroyed handle's streams are kept for the next handle of their own context
only, also where a context is destroyed and another one takes its place.

The contexts other than the primary one are made through the driver API, and
their handles work in memory allocated there (fp32 on the CUDA cores, which
needs no per-device set-up), each giving the primary context's factors bit for
bit.  Run in a process of its own.
"""
import os
import subprocess
import sys

import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

SCRIPT = r"""
import ctypes as C
import numpy as np
import torch
from paper_2608_21607_gb300 import nmd as N
from paper_2608_21607_gb300 import workloads as WL

torch.cuda.init(); torch.zeros(1, device="cuda")
D = C.CDLL("libcuda.so.1")


def ok(st):
    assert st == 0, st


class Mem:   # device memory of the current context
    def __init__(self, n):
        self.n, self.p = n, C.c_uint64()
        ok(D.cuMemAlloc_v2(C.byref(self.p), C.c_size_t(n)))
    def data_ptr(self): return self.p.value
    def numel(self): return self.n
    def element_size(self): return 1
    def free(self): ok(D.cuMemFree_v2(self.p))


S, _, _, _ = WL.planted(300, 200, 4, tau=0.5, seed=0)
W, H = WL.init_factors(300, 200, 4, 0)
opts = N.nmd_default_options()
opts.block_rows = opts.block_cols = 100
opts.precision = N.NMD_SIMT


class Copy:   # a device copy in the current context
    def __init__(self, a):
        self.m = Mem(a.nbytes)
        ok(D.cuMemcpyHtoD_v2(self.m.p, C.c_void_p(a.ctypes.data), C.c_size_t(a.nbytes)))
    def data_ptr(self): return self.m.p.value


def fit(w=None, h_=None):
    ws = Mem(N.nmd_workspace_bytes(S, 4, opts))
    h = N.nmd_create(S, 4, opts, ws, None)
    N.nmd_set_factors(h, W if w is None else w, H if h_ is None else h_, w is not None)
    N.nmd_sweep(h)
    N.nmd_sync(h)
    state = N.nmd_get_state(h, 300, 200, 4)[:4]
    N.nmd_destroy(h)
    ws.free()
    return state


want = fit()
dW, dH = Copy(W), Copy(H)   # in the primary context
for _ in range(3):   # a context that is gone, then one that may be at its address
    ctx = C.c_void_p()
    ok(D.cuCtxCreate_v2(C.byref(ctx), 0, 0))   # made current
    for _ in range(2):
        for x, y in zip(fit() + fit(dW, dH) + fit(Copy(W), Copy(H)), want * 3):
            assert np.array_equal(x, y)
    ok(D.cuCtxPopCurrent_v2(C.byref(C.c_void_p())))
    for x, y in zip(fit() + fit(dW, dH), want * 2):   # in the primary context, the other one alive
        assert np.array_equal(x, y)
    ok(D.cuCtxDestroy_v2(ctx))
    for x, y in zip(fit(), want):
        assert np.array_equal(x, y)
print("contexts ok")
"""


def test_streams_stay_in_their_context():
    require_gpu()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=root, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "PYTHONPATH": root})
    assert r.returncode == 0 and "contexts ok" in r.stdout, r.stdout[-500:] + r.stderr[-2000:]
