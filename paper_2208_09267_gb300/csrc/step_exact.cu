// step_exact.cu -- FP64 step in the canonical evaluation order, and the FP64
// moment / initialisation / population kernels of every storage.
//
// This translation unit is compiled with -fmad=false: no multiply-add is
// fused, so every operation below rounds exactly as written.  The order is
// the canonical one of the method (Sec. 2.2), shared by the FP64 reference:
//   M0 = sum_i f_i and J_a = sum_i xi_ia f_i in ascending i from 0.0;
//   phi_n = phi_ref + (n - n_ref) d_t phi;
//   nb = sum over quadrature axes a of (phi(x+e_a) then phi(x-e_a)) from 0.0;
//   I = varpi_0 phi(x) + varpi_1 nb                           (eq. (quad))
//   rho~ = M0 / I                                             (eq. (density))
//   F_a = (g_a + field_a) + (rho~/3) (0.5 (phi(x+e_a) - phi(x-e_a)))
//                                                             (eq. (pressForce))
//   u_a = (J_a + 0.5 F_a) / M0                                (eq. (velocity))
//   usq = u0 u0 + u1 u1 + u2 u2, uF = u0 F0 + u1 F1 + u2 F2;
//   cu = sum_a xi_ia u_a, cF = sum_a xi_ia F_a from 0.0;
//   f^eq = (w_i M0)(((1 + 3 cu) + (4.5 cu) cu) - 1.5 usq)     (eq. (feq))
//   S = ((1 - 0.5/tau) w_i)((3 (cF - uF)) + (9 cu) cF)        (Guo term)
//   f* = (f + (1/tau)(f^eq - f)) + S                          (eq. (lbe))
// With that order the FP64 result is bit-identical to the reference.
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
  if (L.storage == 1)
    static_cast<float *>(L.pop)[off] = (float)q;
  else
    static_cast<__half *>(L.pop)[off] = __double2half(q);
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
// make_launch_exact).

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

// M0 and J in ascending i
template <class LAT>
__device__ __forceinline__ void sums_exact(const double *f, MacroD &m) {
  constexpr int Q = LAT::Q, D = LAT::D;
  m.M0 = f[0];
#pragma unroll
  for (int i = 1; i < Q; ++i) m.M0 = m.M0 + f[i];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    m.J[a] = 0.0;
    if (a >= D) continue;
    bool any = false;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      if (LAT::c(i, a) == 0) continue;
      const double t = LAT::c(i, a) > 0 ? f[i] : -f[i];
      m.J[a] = any ? m.J[a] + t : t;
      any = true;
    }
  }
}

// rho~, F and u from M0 and J; DRAG: the lattice may carry the drag law
template <class LAT, bool F64, bool DRAG>
__device__ __forceinline__ void macro_from_sums(const LatticeDev &L, long long n, const Coords &C, MacroD &m) {
  constexpr int D = LAT::D;
  const double dn = (double)(n - L.n_eps);
  const double e_c = eps_at<F64>(L, C.at(0, 0, 0), dn);
  double e_p[3], e_m[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (a < D) {
      e_p[a] = eps_at<F64>(L, C.at(a == 0, a == 1, a == 2), dn);
      e_m[a] = eps_at<F64>(L, C.at(-(a == 0), -(a == 1), -(a == 2)), dn);
    } else {
      e_p[a] = e_c;
      e_m[a] = e_c;
    }
  }
  double nb = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (L.quad_axes & (1u << a)) {
      nb = nb + e_p[a];
      nb = nb + e_m[a];
    }
  }
  m.I = L.qw0 * e_c + L.qw1 * nb;
  m.rho = m.M0 / m.I;
  const double pc = m.rho / 3.0;
  const double hpc = 0.5 * pc;  // pc (0.5 (e_p - e_m)) = (0.5 pc) (e_p - e_m) exactly
  const double dnf = (double)(n - L.n_force);
  const long long k = C.at(0, 0, 0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    m.F[a] = 0.0;
    if (a >= D) continue;
    double fext = L.g[a];
    if (L.has_force) fext = fext + force_at<F64>(L, a, k, dnf);
    m.F[a] = fext + hpc * (e_p[a] - e_m[a]);
  }
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

// ---- FP64 step --------------------------------------------------------------

// Write f*_i to its slot of the next step.
template <class LAT, bool ODD>
__device__ __forceinline__ void put_exact(const LatticeDev &L, const Coords &C, int i, int x, int y, int z,
                                          double fstar) {
  const int cx = LAT::c(i, 0), cy = LAT::c(i, 1), cz = LAT::c(i, 2);
  double *pop = static_cast<double *>(L.pop);
  if (!ODD || i == 0 || (L.walls && solid_at(L.walls, x, y, z, cx, cy, cz, L.nx, L.ny, L.nz)))
    pop[(long long)opp_of(i) * L.plane + C.at(0, 0, 0)] = fstar;
  else
    pop[(long long)i * L.plane + C.at(cx, cy, cz)] = fstar;
}

// One thread per cell, cells in linear order over the dense lattice (x
// fastest): a warp is full whatever nx is, which matters where the FP64 pipe
// is the bound (rows of 48 cells as 64 lanes cost a third more).
// EXT: the lattice has the drag law or the closure (a separate instantiation
// keeps the plain step's registers down).
template <class LAT, bool ODD, bool RED, bool EXT>
__global__ void __launch_bounds__(256) step_exact_kernel(const LatticeDev *__restrict__ Lp, int k) {
  constexpr int Q = LAT::Q;
  const LatticeDev &L = *Lp;
  const unsigned nthr = blockDim.x * blockDim.y;
  const long long idx = (long long)blockIdx.x * nthr + threadIdx.y * blockDim.x + threadIdx.x;
  const long long plane_cells = (long long)L.nx * L.ny;
  RedAcc acc;
#pragma unroll
  for (int j = 0; j < kRedWidth; ++j) acc.v[j] = 0.0;
  const bool inside = idx < plane_cells * L.nz;
  const int z = LAT::D == 3 ? (int)(idx / plane_cells) : 0;
  const long long rest = LAT::D == 3 ? idx - z * plane_cells : idx;
  const int y = LAT::D >= 2 ? (int)(rest / L.nx) : 0;
  const int x = (int)(rest - (long long)y * L.nx);
  const bool fluid = inside && !(L.walls && solid_at(L.walls, x, y, z, 0, 0, 0, L.nx, L.ny, L.nz));
  if (fluid) {
    const long long n = L.n + k;
    const Coords C = make_coords(x, y, z, L.nx, L.ny, L.nz, L.nxp);
    const double *pop = static_cast<const double *>(L.pop);
    double f[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const SlotAddr a = slot_of<LAT>(L, C, ODD, i, x, y, z);
      f[i] = pop[(long long)a.slot * L.plane + a.cell];
    }
    MacroD m;
    macro_exact<LAT, true, EXT>(L, n, C, f, m);
    const double usq = dot_d<LAT>(m.u, m.u);
    const double uF = dot_d<LAT>(m.u, m.F);
    if (RED) {
      acc.v[0] += m.M0;
      acc.v[1] += m.J[0] + 0.5 * m.F[0];
      acc.v[2] += m.J[1] + 0.5 * m.F[1];
      acc.v[3] += m.J[2] + 0.5 * m.F[2];
      acc.v[5] += usq;
      if (L.u_prev) {
        float *up = L.u_prev;
        const long long N = L.ncell, c0 = C.at(0, 0, 0);
        if (L.have_prev) {
          const double a = m.u[0] - (double)up[c0], b = m.u[1] - (double)up[N + c0],
                       c = m.u[2] - (double)up[2 * N + c0];
          acc.v[4] += a * a + b * b + c * c;
        }
        up[c0] = (float)m.u[0];
        up[N + c0] = (float)m.u[1];
        up[2 * N + c0] = (float)m.u[2];
      }
      if (!isfinite(m.M0) || !isfinite(usq)) acc.v[6] += 1.0;
      acc.v[7] += m.F[0];
      acc.v[8] += m.F[1];
      acc.v[9] += m.F[2];
    }
    double omega = L.omega, cf = L.cf;
    if (EXT && L.les) {
      // Smagorinsky closure: Pi^neq_ab = sum_i xi_ia xi_ib (f_i - f_i^eq),
      // tau_eff = (tau + sqrt(tau^2 + 18 sqrt(2) C^2 |Pi^neq| / M0)) / 2
      double pi[3][3];
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) pi[a][b] = 0.0;
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const double fneq = f[i] - feq_exact<LAT>(i, m.M0, m.u, usq);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = a; b < 3; ++b) {
            const int cc = LAT::c(i, a) * LAT::c(i, b);
            if (cc != 0) pi[a][b] = cc > 0 ? pi[a][b] + fneq : pi[a][b] - fneq;
          }
      }
      double q2 = 0.0;
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const double v = a <= b ? pi[a][b] : pi[b][a];
          q2 = q2 + v * v;
        }
      const double teff =
          0.5 * (L.tau0 + sqrt(L.tau0 * L.tau0 + 18.0 * sqrt(2.0) * L.les_cs * L.les_cs * sqrt(q2) / m.M0));
      omega = 1.0 / teff;
      cf = 1.0 - 0.5 / teff;
    }
    const double h = 1.5 * usq;
    {
      // rest population: cu = cF = 0
      const double feq = LAT::w(0) * m.M0 * (1.0 - h);
      const double S = cf * LAT::w(0) * (3.0 * (0.0 - uF));
      put_exact<LAT, ODD>(L, C, 0, x, y, z, f[0] + omega * (feq - f[0]) + S);
    }
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
      const double wM = LAT::w(i) * m.M0, cw = cf * LAT::w(i);
      const double cu = dot_c<LAT>(i, m.u), cF = dot_c<LAT>(i, m.F);
      const double t = 3.0 * cu, q = 4.5 * cu * cu, r = 9.0 * cu * cF;
      const double ea = wM * (1.0 + t + q - h), eb = wM * (1.0 - t + q - h);
      const double sa = cw * (3.0 * (cF - uF) + r), sb = cw * (3.0 * (-cF - uF) + r);
      put_exact<LAT, ODD>(L, C, i, x, y, z, f[i] + omega * (ea - f[i]) + sa);
      put_exact<LAT, ODD>(L, C, i + 1, x, y, z, f[i + 1] + omega * (eb - f[i + 1]) + sb);
    }
  }
  if (RED) block_reduce_store(acc, L.partials, blockIdx.x);
}

// ---- moments, initialisation, populations (all storages, FP64 math) ---------

template <class LAT>
__global__ void moments_kernel(const LatticeDev *__restrict__ Lp, double *rho, double *p, double *u,
                               float *rho_f, float *p_f, float *u_f) {
  constexpr int Q = LAT::Q;
  const LatticeDev &L = *Lp;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= L.nx || y >= L.ny) return;
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

template <class LAT, bool F64>
__global__ void init_kernel(const LatticeDev *__restrict__ Lp, const double *p0, const double *u0,
                            int mode) {
  constexpr int Q = LAT::Q, D = LAT::D;
  const LatticeDev &L = *Lp;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= L.nx || y >= L.ny) return;
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

template <class LAT>
__global__ void getpop_kernel(const LatticeDev *__restrict__ Lp, double *out) {
  constexpr int Q = LAT::Q;
  const LatticeDev &L = *Lp;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= L.nx || y >= L.ny) return;
  const Coords C = make_coords(x, y, z, L.nx, L.ny, L.nz, L.nxp);
  const long long kd = ((long long)z * L.ny + y) * L.nx + x;  // dense output index
  const bool solid = L.walls && solid_at(L.walls, x, y, z, 0, 0, 0, L.nx, L.ny, L.nz);
  const bool odd = (L.n & 1) != 0;
#pragma unroll
  for (int i = 0; i < Q; ++i)
    out[kd * Q + i] = solid ? 0.0 : load_f<LAT>(L, slot_of<LAT>(L, C, odd, i, x, y, z), i);
}

// ---- dispatch ----------------------------------------------------------------

template <class LAT, bool EXT>
static cudaError_t launch_exact_ext(const LatticeDev *L_dev, bool odd, int red, int k, const StepLaunch &ls,
                                    cudaStream_t s) {
  if (odd) {
    if (red) step_exact_kernel<LAT, true, true, EXT><<<ls.grid, ls.block, 0, s>>>(L_dev, k);
    else step_exact_kernel<LAT, true, false, EXT><<<ls.grid, ls.block, 0, s>>>(L_dev, k);
  } else {
    if (red) step_exact_kernel<LAT, false, true, EXT><<<ls.grid, ls.block, 0, s>>>(L_dev, k);
    else step_exact_kernel<LAT, false, false, EXT><<<ls.grid, ls.block, 0, s>>>(L_dev, k);
  }
  return cudaGetLastError();
}

template <class LAT>
static cudaError_t launch_exact_lat(const LatticeDev *L_dev, bool ext, bool odd, int red, int k,
                                    const StepLaunch &ls, cudaStream_t s) {
  return ext ? launch_exact_ext<LAT, true>(L_dev, odd, red, k, ls, s)
             : launch_exact_ext<LAT, false>(L_dev, odd, red, k, ls, s);
}

cudaError_t launch_step_exact(const LatticeDev &h, const LatticeDev *L_dev, bool odd, int red, int k,
                              const StepLaunch &ls, cudaStream_t s) {
  const bool ext = h.drag_model || h.les;
  switch (h.lattice) {
    case 0: return launch_exact_lat<D2Q9>(L_dev, ext, odd, red, k, ls, s);
    case 1: return launch_exact_lat<D3Q19>(L_dev, ext, odd, red, k, ls, s);
    case 2: return launch_exact_lat<D3Q27>(L_dev, ext, odd, red, k, ls, s);
    case 3: return launch_exact_lat<D1Q3>(L_dev, ext, odd, red, k, ls, s);
  }
  return cudaErrorInvalidValue;
}

static StepLaunch aux_launch(const LatticeDev &h) { return make_launch(h.nx, h.ny, h.nz, 0, 0); }

cudaError_t launch_moments(const LatticeDev &h, const LatticeDev *L_dev, long long, double *rho,
                           double *p, double *u, float *rho_f, float *p_f, float *u_f,
                           cudaStream_t s) {
  const StepLaunch ls = aux_launch(h);
  switch (h.lattice) {
    case 0: moments_kernel<D2Q9><<<ls.grid, ls.block, 0, s>>>(L_dev, rho, p, u, rho_f, p_f, u_f); break;
    case 1: moments_kernel<D3Q19><<<ls.grid, ls.block, 0, s>>>(L_dev, rho, p, u, rho_f, p_f, u_f); break;
    case 2: moments_kernel<D3Q27><<<ls.grid, ls.block, 0, s>>>(L_dev, rho, p, u, rho_f, p_f, u_f); break;
    case 3: moments_kernel<D1Q3><<<ls.grid, ls.block, 0, s>>>(L_dev, rho, p, u, rho_f, p_f, u_f); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <class LAT>
static void launch_init_lat(const LatticeDev &h, const LatticeDev *L_dev, const double *p0, const double *u0, int mode,
                            const StepLaunch &ls, cudaStream_t s) {
  if (h.storage == 0) init_kernel<LAT, true><<<ls.grid, ls.block, 0, s>>>(L_dev, p0, u0, mode);
  else init_kernel<LAT, false><<<ls.grid, ls.block, 0, s>>>(L_dev, p0, u0, mode);
}

cudaError_t launch_init(const LatticeDev &h, const LatticeDev *L_dev, long long, const double *p0,
                        const double *u0, int mode, cudaStream_t s) {
  const StepLaunch ls = aux_launch(h);
  switch (h.lattice) {
    case 0: launch_init_lat<D2Q9>(h, L_dev, p0, u0, mode, ls, s); break;
    case 1: launch_init_lat<D3Q19>(h, L_dev, p0, u0, mode, ls, s); break;
    case 2: launch_init_lat<D3Q27>(h, L_dev, p0, u0, mode, ls, s); break;
    case 3: launch_init_lat<D1Q3>(h, L_dev, p0, u0, mode, ls, s); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_get_populations(const LatticeDev &h, const LatticeDev *L_dev, long long, double *f,
                                   cudaStream_t s) {
  const StepLaunch ls = aux_launch(h);
  switch (h.lattice) {
    case 0: getpop_kernel<D2Q9><<<ls.grid, ls.block, 0, s>>>(L_dev, f); break;
    case 1: getpop_kernel<D3Q19><<<ls.grid, ls.block, 0, s>>>(L_dev, f); break;
    case 2: getpop_kernel<D3Q27><<<ls.grid, ls.block, 0, s>>>(L_dev, f); break;
    case 3: getpop_kernel<D1Q3><<<ls.grid, ls.block, 0, s>>>(L_dev, f); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace lbm
