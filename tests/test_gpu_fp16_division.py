"""The two-cell update's packed divisions: the operators' results over their
whole range, and the one-cell update where rho0 is outside it."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2208_09267_gb300 import build, lbm

pytestmark = pytest.mark.gpu

CHECK = r"""
#include "step_row.cuh"
using namespace lbm;

__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b) || (isnan(a) && isnan(b)); }
__device__ float with_exponent(int e, unsigned mantissa) { return __uint_as_float((unsigned)(127 + e) << 23 | (mantissa & 0x7fffffu)); }

// every mantissa at exponent e as M0, with hashed and with close mantissas as
// int phi dV from 2^-60 to 1, and as int phi dV itself
__global__ void check(int e, unsigned long long *bad) {
  unsigned long long n = 0;
  auto compare = [&](P2 M0, P2 I) {
    const P2 y = recip2(M0), Is = mul2(I, f2s(kDivScale)), q = quot2(M0, Is, recip2(Is));
    n += !same(lo(y), 1.0f / lo(M0)) + !same(hi(y), 1.0f / hi(M0));
    n += !same(lo(q) * kDivScale, lo(M0) / lo(I)) + !same(hi(q) * kDivScale, hi(M0) / hi(I));
  };
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < (1u << 23); i += gridDim.x * blockDim.x) {
    unsigned h = i * 0x9E3779B9u ^ (unsigned)e;
    for (int j = 0; j < 8; ++j) {
      h = h * 1664525u + 1013904223u;
      const float a = with_exponent(e, i), b = with_exponent(-(int)(h >> 26) % 61, h >> 3), c = with_exponent(0, i + j - 4u);
      compare(f2(j & 1 ? -a : a, a), f2(b, c));
      compare(f2(b, c), f2(with_exponent(-(int)(h & 31u), i), with_exponent(-1, i)));
    }
  }
  atomicAdd(bad, n);
}

extern "C" long long mismatches(int e) {
  unsigned long long *d, h = 0;
  if (cudaMalloc(&d, sizeof(h)) != cudaSuccess) return -1;
  cudaMemset(d, 0, sizeof(h));
  check<<<1216, 256>>>(e, d);
  const cudaError_t err = cudaMemcpy(&h, d, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return err == cudaSuccess ? (long long)h : -1;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("division")
    (d / "check.cu").write_text(CHECK)
    so = str(d / "check.so")
    subprocess.run([build.nvcc()] + build.ARCH + build.COMMON + ["-Xcompiler", "-fvisibility=default", "-shared", "-cudart", "shared", "-o", so, str(d / "check.cu")],
                   check=True, capture_output=True, text=True)
    lib = ctypes.CDLL(so)
    lib.mismatches.restype = ctypes.c_longlong
    return lib


@pytest.mark.parametrize("exponent", [-98, -1, 0, 60])
def test_packed_divisions_give_the_operators_results(harness, exponent):
    assert harness.mismatches(exponent) == 0


@pytest.mark.parametrize("rho0,kind", [
    (8e-39, "slope"),     # M0 is subnormal, its reciprocal finite
    (1.0, "hole"),        # int phi dV is subnormal in one cell, rho~ finite
])
def test_values_at_the_ends_of_the_float_range(rho0, kind):
    """Plain steps, alone (two cells per lane) and in a batch, leave the halves
    of check steps (one cell, operators) where an operand is at the end of the
    float range."""
    shape = (40, 8, 1)
    nx, ny, nz = shape
    flat = np.full(nx * ny, 0.625, dtype=np.float32)
    if kind == "slope":       # halves: the shift is phi itself, nothing is stored of it
        start = phi = np.tile((0.7 + 0.01 * np.sin(2 * np.pi * np.arange(nx) / nx)).astype(np.float16), ny).astype(np.float32)
    else:                     # phi vanishes in one cell of a fluid at rest
        start, phi = flat, flat.copy()
        phi[5 * nx + 17] = 5e-39
    out = {}
    for how in ("check", "plain", "batch"):
        lat = lbm.Lattice("D2Q9", shape, tau=0.6, storage="fp16", rho0=rho0, quad_dim=-1, kernel="row")
        assert lat.row_kernel == (kind == "hole")
        lat.set_epsilon(start)
        lat.init_equilibrium()
        if phi is not start:
            lat.set_epsilon(phi)
        if how == "batch":
            b = lbm.Batch(max_members=1, storage="fp16")
            b.add(lat, 2)
            b.step(2)
            b.close()
        else:
            for _ in range(2):
                lat.step(1, check_every=0 if how == "check" else -1)
        out[how] = lat.populations()
        lat.close()
    assert np.isfinite(out["check"]).all()
    assert np.array_equal(out["plain"], out["check"]) and np.array_equal(out["batch"], out["check"])
