"""The two-cell update's packed divisions: the operators' results for every
operand, and the operators themselves outside the packed ones' range."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2208_09267_gb300 import build, lbm

pytestmark = pytest.mark.gpu

CHECK = r"""
#include "step_row.cuh"
using namespace lbm;

__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b) || (isnan(a) && isnan(b)); }

// every mantissa as M0 and as I at the exponents e of M0, with hashed partners
// of exponents in the packed range, also close to M0 (quotients near 1)
__global__ void check(int e, unsigned long long *bad) {
  unsigned long long n = 0;
  const float i_min = kDivIMin;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < (1u << 23); i += gridDim.x * blockDim.x) {
    unsigned h = i * 0x9E3779B9u ^ (unsigned)e;
    for (int j = 0; j < 8; ++j) {
      const float a = __uint_as_float(((unsigned)e << 23) | i) * (j & 1 ? -1.f : 1.f);
      const float a2 = __uint_as_float(((unsigned)e << 23) | (i ^ 0x2aaaaau));
      h = h * 1664525u + 1013904223u;
      const float b = __uint_as_float((127u - (h >> 27) << 23) + ((h >> 3) & 0x7fffffu));    // 2^-31 .. 2
      const float b2 = __uint_as_float((127u << 23) | ((i + (unsigned)j - 4u) & 0x7fffffu));  // mantissas beside M0's
      P2 y, q;
      inverse_and_quotient2(f2(a, a2), f2(b, b2), i_min, y, q);
      n += !same(lo(y), 1.0f / a) + !same(hi(y), 1.0f / a2) + !same(lo(q), a / b) + !same(hi(q), a2 / b2);
      // the same mantissas as I
      inverse_and_quotient2(f2(b, b2), f2(fabsf(b2), b), i_min, y, q);
      n += !same(lo(y), 1.0f / b) + !same(hi(y), 1.0f / b2) + !same(lo(q), b / b2) + !same(hi(q), b2 / b);
    }
  }
  atomicAdd(bad, n);
}

// operands outside the range: I below the bound, or any with the bound at infinity
__global__ void check_outside(unsigned long long *bad) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  const float a = __uint_as_float(i * 0x9E3779B9u & 0x7fffffffu), b = __uint_as_float(i * 0x85EBCA6Bu & 0x7fffffffu);
  const float c = __uint_as_float((i * 0xC2B2AE35u >> 9) % ((127u - 60u) << 23));                  // below the bound
  unsigned long long n = 0;
  P2 y, q;
  inverse_and_quotient2(f2(a, b), f2(b, a), __int_as_float(0x7f800000), y, q);
  if (!(fminf(a, b) >= __int_as_float(0x7f800000)))
    n += !same(lo(y), 1.0f / a) + !same(hi(y), 1.0f / b) + !same(lo(q), a / b) + !same(hi(q), b / a);
  inverse_and_quotient2(f2(a, b), f2(c, 1.0f), kDivIMin, y, q);
  n += !same(lo(y), 1.0f / a) + !same(hi(y), 1.0f / b) + !same(lo(q), a / c) + !same(hi(q), b / 1.0f);
  atomicAdd(bad, n);
}

extern "C" long long mismatches(int outside) {
  unsigned long long *d, h = 0;
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return -1;
  cudaMemset(d, 0, sizeof(h));
  if (outside) {
    check_outside<<<4096, 256>>>(d);
  } else {
    for (int e = 127 - 98; e <= 127 + 60; e += 79) check<<<1216, 256>>>(e, d);
  }
  const cudaError_t e = cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? (long long)h : -1;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("division")
    (d / "check.cu").write_text(CHECK)
    so = str(d / "check.so")
    subprocess.run([build.nvcc()] + build.ARCH + build.COMMON + ["-shared", "-cudart", "shared", "-o", so, str(d / "check.cu")],
                   check=True, capture_output=True, text=True)
    lib = ctypes.CDLL(so, mode=os.RTLD_LOCAL)
    lib.mismatches.restype = ctypes.c_longlong
    return lib


@pytest.mark.parametrize("outside", [0, 1])
def test_packed_divisions_give_the_operators_results(harness, outside):
    assert harness.mismatches(outside) == 0


@pytest.mark.parametrize("rho0,kind", [
    (8e-39, "slope"),     # M0 is subnormal, its reciprocal finite
    (1.0, "hole"),        # int phi dV is subnormal in one cell, rho~ finite
])
def test_values_at_the_ends_of_the_float_range(rho0, kind):
    """Plain steps (two cells per lane) leave the halves of check steps (one
    cell, operators) where an operand is beyond the packed divisions."""
    shape = (40, 8, 1)
    nx, ny, nz = shape
    flat = np.full(nx * ny, 0.625, dtype=np.float32)
    if kind == "slope":       # halves: the shift is phi itself, nothing is stored of it
        start = phi = np.tile((0.7 + 0.01 * np.sin(2 * np.pi * np.arange(nx) / nx)).astype(np.float16), ny).astype(np.float32)
    else:                     # phi vanishes in one cell of a fluid at rest
        start, phi = flat, flat.copy()
        phi[5 * nx + 17] = 5e-39
    out = []
    for check in (False, True):
        lat = lbm.Lattice("D2Q9", shape, tau=0.6, storage="fp16", rho0=rho0, quad_dim=-1, kernel="row")
        lat.set_epsilon(start)
        lat.init_equilibrium()
        if phi is not start:
            lat.set_epsilon(phi)
        for _ in range(2):
            lat.step(1, check_every=0 if check else -1)
        out.append(lat.populations())
        lat.close()
    assert np.isfinite(out[1]).all()
    assert np.array_equal(*out)
