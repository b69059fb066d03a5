"""Calls in several CUDA contexts of one process, one after the other, and after
the primary context has been reset.

What the library keeps between calls has to hold in each of them: the stepper
kernels' raised shared-memory limit (launches above 48 KB: 512 threads per block,
or many sets), the memory pool (which belongs to the device) and the fixed
scratch of the no-allocation entry.  The contexts are made, reset and destroyed
through the driver, in a child process that holds no other.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r'''
import ctypes, types
from paper_2206_11234_gb300 import native as nat, workloads as W
cu = ctypes.CDLL("libcuda.so.1")
NULL_STREAM = types.SimpleNamespace(cuda_stream=0)  # torch's current stream would bring torch's context


def ok(rc):
    assert rc == 0, rc


ok(cu.cuInit(0))
dev = ctypes.c_int()
ok(cu.cuDeviceGet(ctypes.byref(dev), 0))


def malloc(nbytes):
    p = ctypes.c_uint64()
    ok(cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(nbytes)))
    return p


def host(p, nbytes):
    b = ctypes.create_string_buffer(nbytes)
    ok(cu.cuMemcpyDtoH_v2(b, p, ctypes.c_size_t(nbytes)))
    return b.raw


def in_new_context(body):
    ctx = ctypes.c_void_p()
    ok(cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, dev))
    out = body()
    ok(cu.cuCtxDestroy_v2(ctx))
    return out


lib = nat.lib
noalloc = lib.fpt_simulate_batch_noalloc
noalloc.argtypes = [ctypes.POINTER(nat.FptParams), ctypes.POINTER(nat.FptSet), ctypes.c_int32, ctypes.c_uint64,
                    ctypes.c_void_p, ctypes.c_void_p]


def records(entry, n_sets, each, **kw):
    specs = [W.SetSpec(phi_in=2.0, m=1.0, b=0.5, dN=2e-3, n_max=1.0, n_traj=each, set_id=i) for i in range(n_sets)]
    n = n_sets * each
    N, lw = malloc(8 * n), malloc(8 * n)
    p = nat.make_params(m=1.0, n_max=1.0, stream=NULL_STREAM, **kw)
    args = (ctypes.byref(p), nat.make_sets(specs), n_sets, 7, N.value, lw.value)
    rc = noalloc(*args) if entry == "noalloc" else lib.fpt_simulate_batch(*args, None, None)
    assert rc == nat.FPT_OK, (entry, kw, lib.fpt_last_error())
    return host(N, 8 * n) + host(lw, 8 * n)
'''


BODY = CHILD + r'''
import numpy as np


def body():
    out = [records("noalloc", 2, 2000, precision="f32_kahan", block_dim=512),
           records("noalloc", 48, 20, precision="f64"),
           records("noalloc", 48, 20, precision="f64", block_dim=512),
           records("batch", 64, 100, precision="f32_f64acc", block_dim=256)]
    # the network's value, whose status word comes from the pool
    w = nat.mlp_pack(W.mlp_params(seed=3, gain=1.0, out_scale=0.5), (2.0, 1.0, 1.0, 1.0), device="cpu")
    n = 300
    pw, x, b = malloc(w.numel()), malloc(4 * n), malloc(4 * n)
    ok(cu.cuMemcpyHtoD_v2(pw, ctypes.c_void_p(w.data_ptr()), ctypes.c_size_t(w.numel())))
    rows = np.linspace(1.5, 3.0, n, dtype=np.float32)
    ok(cu.cuMemcpyHtoD_v2(x, rows.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(4 * n)))
    rc = lib.fpt_mlp_forward(pw.value, x.value, x.value, n, b.value, None)
    assert rc == nat.FPT_OK, lib.fpt_last_error()
    return out + [host(b, 4 * n)]


first = in_new_context(body)
assert len(set(first[0])) > 100 and len(set(first[-1])) > 100
for _ in range(2):
    assert in_new_context(body) == first
for _ in range(2):  # the primary context, reset between
    ctx = ctypes.c_void_p()
    ok(cu.cuDevicePrimaryCtxRetain(ctypes.byref(ctx), dev))
    ok(cu.cuCtxSetCurrent(ctx))
    assert body() == first
    ok(cu.cuDevicePrimaryCtxReset_v2(dev))
print("same results")
'''


def test_new_contexts_and_a_reset():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", BODY], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "same results" in r.stdout
