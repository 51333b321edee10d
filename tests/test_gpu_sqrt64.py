"""The square root of the FP64 flux (sqrt64.cuh) against the correctly rounded one: equal outside the range of its
own iteration (zeros, subnormal and tiny numbers, negative, infinite and NaN arguments) and within one unit in
the last place inside it, where only roots next to the midpoint of two numbers may differ at all (an estimate
good to 2^-20 leaves 2^-27 of a unit: less than one of 10^4 random arguments)."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np
import pytest

import paper_2312_17042_gb300 as package
from paper_2312_17042_gb300 import build
from tests.test_gpu_parity import _native

pytestmark = pytest.mark.gpu

SOURCE = """
#include "sqrt64.cuh"
__global__ void roots(const double *x, double *y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = cteno::sqrt64(x[i]);
}
extern "C" int run(const double *x, double *y, int n) {
  roots<<<(n + 255) / 256, 256>>>(x, y, n);
  return cudaDeviceSynchronize();
}
"""


def _roots(tmp_path, x):
    import torch
    (tmp_path / "roots.cu").write_text(SOURCE)
    lib = str(tmp_path / "roots.so")
    subprocess.run(["nvcc", build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(os.path.dirname(package.__file__), "csrc"), str(tmp_path / "roots.cu"), "-o", lib],
                   check=True)
    a = torch.from_numpy(x).cuda()
    b = torch.empty_like(a)
    assert ctypes.CDLL(lib).run(ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(b.data_ptr()), ctypes.c_int(x.size)) == 0
    return b.cpu().numpy()


def test_against_the_correctly_rounded_root(tmp_path):
    _native()
    rng = np.random.default_rng(1)
    n = 1 << 20
    random = np.ldexp(rng.uniform(1, 2, n), rng.integers(-1022, 1024, n))
    powers = np.ldexp(1.0, np.arange(-1022, 1024))
    squares = rng.integers(1, 1 << 26, 1 << 16).astype(float) ** 2
    edges = np.concatenate([powers, squares])
    edges = np.concatenate([edges, np.nextafter(edges, 0), np.nextafter(edges, np.inf)])
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -np.nan, -1.0, -5e-324, 5e-324, 2.0 ** -1023, np.finfo(float).max])
    x = np.concatenate([random, edges, special])
    y = _roots(tmp_path, x)
    with np.errstate(invalid="ignore"):
        ref = np.sqrt(x)
    own = (x >= 2.0 ** -959) & np.isfinite(x)
    assert np.array_equal(y[~own], ref[~own], equal_nan=True)
    assert np.array_equal(np.signbit(y[x == 0]), np.signbit(ref[x == 0]))
    assert np.all(np.abs(y[own].view(np.int64) - ref[own].view(np.int64)) <= 1)
    assert np.count_nonzero(y[:n] != ref[:n]) <= 1e-4 * n
