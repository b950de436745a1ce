"""The coarse CG's scalars (csrc/cg_scalar.cuh) against IEEE arithmetic: the
reciprocal over its range, the power of two that brings a load into range, and
the stopping test against the square root.

The reciprocal's bound: the hardware's approximation is good to 2^-20, so the
third-order step leaves 2^-60 and the rounding of its last operation, half a
unit in the last place; the correctly rounded reciprocal is then the same or a
neighbour."""

import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cuda_runtime.h>
#include "cg_scalar.cuh"
__global__ void k(int what, int n, const double* a, const double* b, double* out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  if (what == 0) out[q] = cg_recip(b[q]);
  if (what == 1) out[q] = cg_in_range(a[q]) ? 1.0 : cg_shift(cg_exponent(b[q]));
  if (what == 2) out[q] = cg_above(a[q], cg_test(b[q])) ? 1.0 : 0.0;
}
extern "C" int run(int what, int n, const double* a, const double* b, double* out) {
  k<<<(n + 255) / 256, 256>>>(what, n, a, b, out);
  cudaError_t e = cudaDeviceSynchronize();
  return (int)(e ? e : cudaGetLastError());
}
"""


@pytest.fixture(scope="module")
def scalar(tmp_path_factory):
    import torch
    import importlib
    B = importlib.import_module("paper_1506_06185_gb300.build")
    d = tmp_path_factory.mktemp("cg_scalar")
    (d / "t.cu").write_text(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC,
                    str(d / "t.cu"), "-o", str(d / "t.so")], check=True)
    lib = ctypes.CDLL(os.path.join(str(d), "t.so"))
    lib.run.argtypes = [ctypes.c_int, ctypes.c_int] + [ctypes.c_void_p] * 3

    def call(what, a, b):
        ta, tb = (torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).cuda() for v in (a, b))
        out = torch.empty_like(tb)
        torch.cuda.synchronize()
        assert lib.run(what, tb.numel(), ta.data_ptr(), tb.data_ptr(), out.data_ptr()) == 0
        return out.cpu().numpy()
    return call


def _values(exponents, n, seed):
    """Random and extreme mantissas at every biased exponent given."""
    r = np.random.default_rng(seed)
    m = np.concatenate([r.integers(0, 1 << 52, n), [0, 1, (1 << 52) - 1, (1 << 52) - 2]]).astype(np.uint64)
    return ((np.asarray(exponents, dtype=np.uint64) << np.uint64(52))[:, None] | m[None]).reshape(-1).view(np.float64)


def test_reciprocal(scalar):
    b = _values(np.arange(2, 2044), 500, 1)               # 2^-1021 .. 2^1021
    got, want = scalar(0, b, b), 1.0 / b
    assert (np.abs(got.view(np.int64) - want.view(np.int64)) <= 1).all()
    assert np.array_equal(scalar(0, b, -b), -got)


def test_shift(scalar):
    b = _values(np.arange(0, 2047), 20, 2)
    up = scalar(1, np.zeros_like(b), b)
    assert (np.frexp(up)[0] == 0.5).all() and np.isfinite(1.0 / up).all() and (1.0 / (1.0 / up) == up).all()
    e = b.view(np.uint64) >> np.uint64(52)
    mid = (e >= 1) & (e <= 2023)
    assert ((b * up >= 1) & (b * up < 2))[mid].all()
    assert (b * up < 2.0 ** 24).all()                     # the largest numbers
    assert (scalar(1, np.zeros(3), [math.inf, -math.inf, math.nan]) == 1.0).all()
    # a load is left alone where b.b lies in 2^-400 .. 2^401
    bb = np.ldexp(1.0, [-1074, -401, -400, 0, 400, 401, 1023])
    assert ((scalar(1, bb, np.full(7, 8.0)) == 1.0) == [False, False, True, True, True, False, False]).all()
    assert (scalar(1, [0.0, math.inf, math.nan], np.full(3, 8.0)) == 0.125).all()


def test_stopping_test(scalar):
    r = np.random.default_rng(6)
    thr = np.concatenate([np.ldexp(r.uniform(0.5, 1, 20000), r.integers(-600, 500, 20000)), np.full(7, 0.0),
                          np.full(7, 1e-3)])
    rr = thr * thr * (1 + np.concatenate([r.choice([-1, 1], 10000) * 10.0 ** r.uniform(-17, 1, 10000),
                                          r.integers(-6, 7, 10000) * 2.0 ** -53, np.zeros(14)]))
    rr = np.abs(rr)
    rr[-14:] = np.tile([0.0, 5e-324, 1e-300, 1.0, 1e300, math.inf, math.nan], 2)
    assert np.array_equal(scalar(2, rr, thr) != 0.0, np.sqrt(rr) > thr)
