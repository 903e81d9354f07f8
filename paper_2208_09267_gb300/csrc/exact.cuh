// exact.cuh -- one cell's moments, initial state and macroscopic quantities in
// FP64 arithmetic, in the canonical order that step_exact.cu states.
//
// step_exact.cu includes it with -fmad=false, where the results are
// bit-identical to the reference; fields_ff.cu takes the cells whose values
// leave the range of its float-float arithmetic from here.
#pragma once

#include <cuda_fp16.h>

#include "internal.h"
#include "lattice.cuh"
#include "step_fast.cuh"

namespace lbm {

// Address (slot, cell) holding f_i(x, n) at the parity of n, AA pattern.
struct SlotAddr {
  int slot;
  long long cell;
};

template <class LAT>
__device__ __forceinline__ SlotAddr slot_of(const LatticeDev &L, const Coords &C, bool odd_layout,
                                            int i, int x, int y, int z) {
  SlotAddr a;
  const int cx = LAT::c(i, 0), cy = LAT::c(i, 1), cz = LAT::c(i, 2);
  if (!odd_layout || i == 0) {
    a.slot = i;
    a.cell = C.at(0, 0, 0);
  } else if (L.walls && solid_at(L.walls, x, y, z, -cx, -cy, -cz, L.nx, L.ny, L.nz)) {
    a.slot = i;
    a.cell = C.at(0, 0, 0);
  } else {
    a.slot = opp_of(i);
    a.cell = C.at(-cx, -cy, -cz);
  }
  return a;
}

// Read f_i(x, n) of any storage as a double.
template <class LAT>
__device__ __forceinline__ double load_f(const LatticeDev &L, const SlotAddr &a, int i) {
  const long long off = (long long)a.slot * L.plane + a.cell;
  if (L.storage == 0) return static_cast<const double *>(L.pop)[off];
  double q = L.storage == 1 ? (double)static_cast<const float *>(L.pop)[off]
                            : (double)__half2float(static_cast<const __half *>(L.pop)[off]);
  const double s = L.rho0 * (double)__half2float(L.sig_rd[a.cell]);
  return LAT::w(i) * (s + q * (double)L.inv_scale);
}

// Write a stored value of any storage.
__device__ __forceinline__ void put_stored(const LatticeDev &L, const SlotAddr &a, double q) {
  const long long off = (long long)a.slot * L.plane + a.cell;
  if (L.storage == 0)
    static_cast<double *>(L.pop)[off] = q;
  else if (L.storage == 1)
    static_cast<float *>(L.pop)[off] = (float)q;
  else
    static_cast<__half *>(L.pop)[off] = __double2half(q);
}

// Write f_i to a slot of any storage (encoding against sigma_wr).
template <class LAT>
__device__ __forceinline__ void store_f(const LatticeDev &L, int slot, long long cell, int i, double f) {
  const long long off = (long long)slot * L.plane + cell;
  if (L.storage == 0) {
    static_cast<double *>(L.pop)[off] = f;
    return;
  }
  const double s = L.rho0 * (double)__half2float(L.sig_wr[cell]);
  const double q = (f / LAT::w(i) - s) * (double)L.scale;
  put_stored(L, SlotAddr{slot, cell}, q);
}

struct MacroD {
  double M0, J[3], I, rho, F[3], u[3];
};

// phi at time n of the FP64 fields (F64) or of the FP32 fields of the other
// storages, in double.
template <bool F64>
__device__ __forceinline__ double eps_at(const LatticeDev &L, long long m, double dn) {
  if (F64) {
    const double *e = static_cast<const double *>(L.eps);
    if (L.has_deps) return e[m] + dn * static_cast<const double *>(L.deps)[m];
    return e[m];
  }
  const float *e = static_cast<const float *>(L.eps);
  if (L.has_deps) return (double)e[m] + dn * (double)static_cast<const float *>(L.deps)[m];
  return (double)e[m];
}

template <bool F64>
__device__ __forceinline__ double force_at(const LatticeDev &L, int a, long long k, double dnf) {
  const long long off = (long long)a * L.ncell + k;
  if (F64) {
    double fa = static_cast<const double *>(L.force)[off];
    if (L.has_dforce) fa = fa + dnf * static_cast<const double *>(L.dforce)[off];
    return fa;
  }
  double fa = (double)static_cast<const float *>(L.force)[off];
  if (L.has_dforce) fa = fa + dnf * (double)static_cast<const float *>(L.dforce)[off];
  return fa;
}

// What bounds the FP64 kernels: the FP64 pipe takes 64 clocks for a warp
// instruction on each quarter of an SM, 19 with all four busy (measured; the
// lanes in use do not matter), a 64th of the FP32 rate, so every operation
// below counts and loads do not.  The operations are
// those of the canonical order with the ones that cannot change a result
// left out: terms with a zero velocity component (x + 0 y = x for finite
// y), products by +-1 and +-1/2 (exact, so they move freely; J + F/2 is one
// FMA), and what a population shares with its opposite (c u and c F change
// sign exactly, (4.5 cu) cu and (9 cu) cF do not).  About 240 operations per
// D2Q9 cell, 430 D3Q19, 600 D3Q27: a 48^3 D3Q27 step 138 us (before 240), a
// 64 x 64 D2Q9 step 9.6 us (26, most of it from the smaller blocks of
// make_launch_exact; 6.1 with four warps to 32 cells, step_exact.cu).

// sum over the velocities of one set of c_ia v_a, terms in ascending a
template <class LAT>
__device__ __forceinline__ double dot_c(int i, const double *v) {
  double s = 0.0;
  bool any = false;
#pragma unroll
  for (int a = 0; a < LAT::D; ++a) {
    if (LAT::c(i, a) == 0) continue;
    const double t = LAT::c(i, a) > 0 ? v[a] : -v[a];
    s = any ? s + t : t;
    any = true;
  }
  return s;
}

// M0, and the momentum along axis a, in ascending i
template <class LAT>
__device__ __forceinline__ double sum_m0(const double *f) {
  double s = f[0];
#pragma unroll
  for (int i = 1; i < LAT::Q; ++i) s = s + f[i];
  return s;
}

template <class LAT>
__device__ __forceinline__ double sum_j(const double *f, int a) {
  double s = 0.0;
  bool any = false;
#pragma unroll
  for (int i = 1; i < LAT::Q; ++i) {
    if (LAT::c(i, a) == 0) continue;
    const double t = LAT::c(i, a) > 0 ? f[i] : -f[i];
    s = any ? s + t : t;
    any = true;
  }
  return s;
}

template <class LAT>
__device__ __forceinline__ void sums_exact(const double *f, MacroD &m) {
  m.M0 = sum_m0<LAT>(f);
#pragma unroll
  for (int a = 0; a < 3; ++a) m.J[a] = a < LAT::D ? sum_j<LAT>(f, a) : 0.0;
}

// phi at time n on the cell and its face neighbours
template <class LAT, bool F64>
__device__ __forceinline__ void phi_stencil(const LatticeDev &L, long long n, const Coords &C, double &e_c,
                                            double *e_p, double *e_m) {
  const double dn = (double)(n - L.n_eps);
  e_c = eps_at<F64>(L, C.at(0, 0, 0), dn);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (a < LAT::D) {
      e_p[a] = eps_at<F64>(L, C.at(a == 0, a == 1, a == 2), dn);
      e_m[a] = eps_at<F64>(L, C.at(-(a == 0), -(a == 1), -(a == 2)), dn);
    } else {
      e_p[a] = e_c;
      e_m[a] = e_c;
    }
  }
}

// eq. (quad)
__device__ __forceinline__ double quad_exact(const LatticeDev &L, double e_c, const double *e_p, const double *e_m) {
  double nb = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (L.quad_axes & (1u << a)) {
      nb = nb + e_p[a];
      nb = nb + e_m[a];
    }
  }
  return L.qw0 * e_c + L.qw1 * nb;
}

// force along axis a
template <bool F64>
__device__ __forceinline__ double force_exact(const LatticeDev &L, long long n, const Coords &C, int a, double rho,
                                              double e_p, double e_m) {
  const double pc = rho / 3.0;
  const double hpc = 0.5 * pc;  // pc (0.5 (e_p - e_m)) = (0.5 pc) (e_p - e_m) exactly
  double fext = L.g[a];
  if (L.has_force) fext = fext + force_at<F64>(L, a, C.at(0, 0, 0), (double)(n - L.n_force));
  return fext + hpc * (e_p - e_m);
}

// rho~, F and u from M0 and J; DRAG: the lattice may carry the drag law
template <class LAT, bool F64, bool DRAG>
__device__ __forceinline__ void macro_from_sums(const LatticeDev &L, long long n, const Coords &C, MacroD &m) {
  constexpr int D = LAT::D;
  double e_c, e_p[3], e_m[3];
  phi_stencil<LAT, F64>(L, n, C, e_c, e_p, e_m);
  m.I = quad_exact(L, e_c, e_p, e_m);
  m.rho = m.M0 / m.I;
#pragma unroll
  for (int a = 0; a < 3; ++a) m.F[a] = a < D ? force_exact<F64>(L, n, C, a, m.rho, e_p[a], e_m[a]) : 0.0;
  if (!DRAG || !L.drag_model) {
#pragma unroll
    for (int a = 0; a < 3; ++a) m.u[a] = a < D ? __fma_rn(0.5, m.F[a], m.J[a]) / m.M0 : 0.0;
    return;
  }
  // phase-interaction drag F_D = -(b_lin + b_q |u|) u (Ergun-type law of a
  // fixed bed, Sec. 2.2's force sum), implicit in eq. (velocity): with
  // b = J + F/2 the speed s = |u| is the positive root of
  // (b_q/2) s^2 + (M0 + b_lin/2) s - |b| = 0, u = b / (M0 + b_lin/2 + b_q s/2)
  const double one_m = 1.0 - e_c;
  const double nu = (L.tau0 - 0.5) / 3.0;
  const double blin = m.rho * L.drag_c1 * one_m * one_m * nu / (e_c * L.drag_d * L.drag_d);
  const double bq = m.rho * L.drag_c2 * one_m / L.drag_d;
  double b[3], bn = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    b[a] = m.J[a] + 0.5 * m.F[a];
    bn = bn + b[a] * b[a];
  }
  bn = sqrt(bn);
  const double A = m.M0 + 0.5 * blin;
  const double sp = 2.0 * bn / (A + sqrt(A * A + 2.0 * bq * bn));
  const double den = A + 0.5 * bq * sp;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    m.u[a] = b[a] / den;
    const double fd = (blin + bq * sp) * m.u[a];
    m.F[a] = (a < D) ? m.F[a] - fd : 0.0;
  }
}

template <class LAT, bool F64, bool DRAG = true>
__device__ __forceinline__ void macro_exact(const LatticeDev &L, long long n, const Coords &C, const double *f,
                                            MacroD &m) {
  sums_exact<LAT>(f, m);
  macro_from_sums<LAT, F64, DRAG>(L, n, C, m);
}

// a . b over the lattice's axes, ascending
template <class LAT>
__device__ __forceinline__ double dot_d(const double *a, const double *b) {
  double s = a[0] * b[0];
#pragma unroll
  for (int k = 1; k < LAT::D; ++k) s = s + a[k] * b[k];
  return s;
}

template <class LAT>
__device__ __forceinline__ double feq_exact(int i, double M0, const double *u, double usq) {
  const double cu = dot_c<LAT>(i, u);
  return LAT::w(i) * M0 * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq);
}

// Moments of one cell at the device-side time (any output may be null).
template <class LAT>
__device__ __forceinline__ void moments_cell(const LatticeDev &L, int x, int y, int z, double *rho, double *p,
                                             double *u, float *rho_f, float *p_f, float *u_f) {
  constexpr int Q = LAT::Q;
  const Coords C = make_coords(x, y, z, L.nx, L.ny, L.nz, L.nxp);
  // outputs are dense: index (z*ny + y)*nx + x, N = nx*ny*nz
  const long long k = ((long long)z * L.ny + y) * L.nx + x;
  const long long N = (long long)L.nx * L.ny * L.nz;
  const bool odd = (L.n & 1) != 0;
  if (L.walls && solid_at(L.walls, x, y, z, 0, 0, 0, L.nx, L.ny, L.nz)) {
    if (rho) rho[k] = 0.0;
    if (p) p[k] = 0.0;
    if (rho_f) rho_f[k] = 0.f;
    if (p_f) p_f[k] = 0.f;
    for (int a = 0; a < 3; ++a) {
      if (u) u[a * N + k] = 0.0;
      if (u_f) u_f[a * N + k] = 0.f;
    }
    return;
  }
  double f[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = load_f<LAT>(L, slot_of<LAT>(L, C, odd, i, x, y, z), i);
  MacroD m;
  if (L.storage == 0) macro_exact<LAT, true>(L, L.n, C, f, m);
  else macro_exact<LAT, false>(L, L.n, C, f, m);
  const double pv = (m.rho - L.rho0) / 3.0;
  if (rho) rho[k] = m.rho;
  if (p) p[k] = pv;
  if (rho_f) rho_f[k] = (float)m.rho;
  if (p_f) p_f[k] = (float)pv;
  for (int a = 0; a < 3; ++a) {
    if (u) u[a * N + k] = m.u[a];
    if (u_f) u_f[a * N + k] = (float)m.u[a];
  }
}

// Initial populations of one cell (mode bits as lbm_vanse_init_equilibrium).
template <class LAT, bool F64>
__device__ __forceinline__ void init_cell(const LatticeDev &L, int x, int y, int z, const double *p0,
                                          const double *u0, int mode) {
  constexpr int Q = LAT::Q, D = LAT::D;
  if (L.walls && solid_at(L.walls, x, y, z, 0, 0, 0, L.nx, L.ny, L.nz)) return;
  const Coords C = make_coords(x, y, z, L.nx, L.ny, L.nz, L.nxp);
  const long long k = C.at(0, 0, 0);
  // p0, u0 are dense arrays: index (z*ny + y)*nx + x, N = nx*ny*nz
  const long long kd = ((long long)z * L.ny + y) * L.nx + x;
  const long long N = (long long)L.nx * L.ny * L.nz;
  const long long n = L.n;
  const bool odd = (n & 1) != 0;
  double u[3] = {0.0, 0.0, 0.0};
  if (u0)
    for (int a = 0; a < D; ++a) u[a] = u0[a * N + kd];
  double usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const double rt = L.rho0 + (p0 ? 3.0 * p0[kd] : 0.0);
  const double dn = (double)(n - L.n_eps);
  double mass;
  if (mode & 1) {
    double nb = 0.0;
    for (int a = 0; a < 3; ++a) {
      if (L.quad_axes & (1u << a)) {
        nb = nb + eps_at<F64>(L, C.at(a == 0, a == 1, a == 2), dn);
        nb = nb + eps_at<F64>(L, C.at(-(a == 0), -(a == 1), -(a == 2)), dn);
      }
    }
    mass = rt * (L.qw0 * eps_at<F64>(L, k, dn) + L.qw1 * nb);
  } else {
    mass = rt * eps_at<F64>(L, k, dn);
  }
  if (!u0 && !(mode & 2)) {
    // u = 0: f_i = w_i m, one value per weight class (FP32/FP16: the value
    // stored against a shift; at even n every slot has the cell's own), so
    // three divisions a cell instead of one per population: 256^3 D3Q19 FP16
    // 2.6 ms (before 14.5)
    const double s_own = F64 ? 0.0 : L.rho0 * (double)__half2float(L.sig_wr[k]);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int first = c == 0 ? 0 : (c == 1 ? 1 : (c == 2 ? 2 * D + 1 : 19));
      const int last = c == 0 ? 0 : (c == 1 ? 2 * D : (c == 2 ? (Q < 19 ? Q - 1 : 18) : Q - 1));
      if (first > last) continue;
      const double f = LAT::w(first) * mass;
      const double d = F64 ? f : f / LAT::w(first);
      const double q_own = F64 ? f : (d - s_own) * (double)L.scale;
#pragma unroll
      for (int i = first; i <= last; ++i) {
        const SlotAddr a = slot_of<LAT>(L, C, odd, i, x, y, z);
        double q = q_own;
        if (!F64 && odd) q = (d - L.rho0 * (double)__half2float(L.sig_wr[a.cell])) * (double)L.scale;
        put_stored(L, a, q);
      }
    }
    return;
  }
  double f[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = feq_exact<LAT>(i, mass, u, usq);
  if (mode & 2) {
    MacroD m;
    macro_exact<LAT, F64>(L, n, C, f, m);
    for (int a = 0; a < 3; ++a) u[a] = u[a] - 0.5 * m.F[a] / m.M0;
    usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = feq_exact<LAT>(i, mass, u, usq);
  }
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const SlotAddr a = slot_of<LAT>(L, C, odd, i, x, y, z);
    store_f<LAT>(L, a.slot, a.cell, i, f[i]);
  }
}

}  // namespace lbm
