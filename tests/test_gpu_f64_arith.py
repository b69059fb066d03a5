"""The binary64 reciprocal, square root and logarithm of the reference stepper (csrc/rng64.cuh) by
themselves, against arithmetic of more bits.

A small library of three loops over them is compiled here, without contraction, as
the stepper is.  Bounds, in units in the last place (ulp, 2^-52 of the power of two
below):
  reciprocal: the seed errs by at most 2^-19 (about 2^-20 in fact), the third-order step
    leaves its cube, 2^-57, and rounds once: 0.5 + 2^-4 ulp;
  root: the same once, and half of g's own rounding (2^-54 of the result, at most half
    an ulp): 1 + 2^-4 ulp;
  radius: half the logarithm's relative error (2.5 x 2^-52, test_f64_tables.py) and the root's
    (2^-53 + 2^-54): below 4.5e-16 relative.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2206_11234_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
#include "rng64.cuh"
__global__ void eval(int what, const double* x, const unsigned* w, double* y, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        y[i] = what == 0   ? fpt::reciprocal(x[i])
               : what == 1 ? fpt::root(x[i])
               : what == 2 ? fpt::minus_two_ln(w[i])
                           : fpt::root(fpt::minus_two_ln(w[i]));
}
extern "C" int run(int what, const double* x, const unsigned* w, double* y, int n) {
    eval<<<64, 256>>>(what, x, w, y, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def device(cuda_device, tmp_path_factory):
    import torch
    build.build()  # writes the tables
    d = tmp_path_factory.mktemp("arith")
    src, lib = d / "arith.cu", d / "libarith.so"
    src.write_text(SOURCE)
    for name, text in (("f64_tables.inc", build.f64_tables()),):
        (d / name).write_text(text)
    subprocess.run([build.nvcc(), *build.ARCH, *build.COMMON, "-I" + str(d), "-fmad=false", "-shared", str(src), "-o", str(lib)],
                   check=True, capture_output=True, text=True)
    f = ctypes.CDLL(os.fspath(lib)).run
    f.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]

    def call(what, v):
        y = torch.empty(v.size, dtype=torch.float64, device="cuda")
        t = torch.from_numpy(v.view(np.int32) if v.dtype == np.uint32 else v).cuda()
        torch.cuda.synchronize()
        args = (None, t.data_ptr()) if v.dtype == np.uint32 else (t.data_ptr(), None)
        assert f(what, *args, y.data_ptr(), v.size) == 0
        return y.cpu().numpy()

    return call


def ulps(got, exact):
    return np.abs((got - exact) / np.spacing(np.abs(got))).astype(np.float64)


def mantissas(rng):
    k = np.arange(4096)
    return np.concatenate([1.0 + k / 4096, np.nextafter(1.0 + k / 4096, 0), 1.0 + (k + 0.5) / 4096, np.nextafter(2.0 - k * 2.0 ** -40, 0),
                           1.0 + rng.random(1 << 18)])


def test_reciprocal(device):
    rng = np.random.default_rng(1)
    m = mantissas(rng)
    x = np.concatenate([m, np.ldexp(m, rng.integers(-900, 900, m.size)), -m])
    got = device(0, x)
    assert np.finfo(np.longdouble).nmant >= 63
    assert ulps(got, 1 / x.astype(np.longdouble)).max() <= 0.5 + 2.0 ** -4


def test_root(device):
    rng = np.random.default_rng(2)
    m = mantissas(rng)
    # -2 ln u0 lies between 2.3e-10 and 46
    x = np.concatenate([m, 2 * m, np.ldexp(m, rng.integers(-33, 6, m.size)), 46 * rng.random(1 << 18) + 1e-12])
    assert ulps(device(1, x), np.sqrt(x.astype(np.longdouble))).max() <= 1.0 + 2.0 ** -4


def test_logarithm_and_radius(device):
    rng = np.random.default_rng(3)
    w = np.concatenate([np.arange(4096), 2 ** 32 - 1 - np.arange(4096), rng.integers(0, 2 ** 32, 1 << 19)] +
                       [np.clip(2 ** p + np.arange(-3, 4), 0, 2 ** 32 - 1) for p in range(1, 32)]).astype(np.uint32)
    exact = -2 * np.log((w.astype(np.longdouble) + np.longdouble(0.5)) / np.longdouble(2 ** 32))
    rel = lambda got, ref: np.abs((got - ref) / ref).astype(np.float64)  # noqa: E731
    assert rel(device(2, w), exact).max() <= 2.5 * 2.0 ** -52
    r = rel(device(3, w), np.sqrt(exact))
    assert r.max() <= 4.5e-16 and r.mean() <= 1e-16, (r.max(), r.mean())
