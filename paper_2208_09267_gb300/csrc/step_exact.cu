// step_exact.cu -- FP64 step in the canonical evaluation order, the FP64 and
// FP16 initialisation, and the moment and population kernels in FP64
// arithmetic (single-precision moments, FP32 initial state: fields_ff.cu).
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
#include "exact.cuh"

namespace lbm {

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

// Collide and stream the rest population (cu = cF = 0).
template <class LAT, bool ODD>
__device__ __forceinline__ void collide_rest(const LatticeDev &L, const Coords &C, int x, int y, int z,
                                             const MacroD &m, double uF, double h, double omega, double cf, double f) {
  const double feq = LAT::w(0) * m.M0 * (1.0 - h);
  const double S = cf * LAT::w(0) * (3.0 * (0.0 - uF));
  put_exact<LAT, ODD>(L, C, 0, x, y, z, f + omega * (feq - f) + S);
}

// Collide and stream the opposite populations i and i + 1 (values fa, fb).
template <class LAT, bool ODD>
__device__ __forceinline__ void collide_pair(const LatticeDev &L, const Coords &C, int i, int x, int y, int z,
                                             const MacroD &m, double uF, double h, double omega, double cf, double fa,
                                             double fb) {
  const double wM = LAT::w(i) * m.M0, cw = cf * LAT::w(i);
  const double cu = dot_c<LAT>(i, m.u), cF = dot_c<LAT>(i, m.F);
  const double t = 3.0 * cu, q = 4.5 * cu * cu, r = 9.0 * cu * cF;
  const double ea = wM * (1.0 + t + q - h), eb = wM * (1.0 - t + q - h);
  const double sa = cw * (3.0 * (cF - uF) + r), sb = cw * (3.0 * (-cF - uF) + r);
  put_exact<LAT, ODD>(L, C, i, x, y, z, fa + omega * (ea - fa) + sa);
  put_exact<LAT, ODD>(L, C, i + 1, x, y, z, fb + omega * (eb - fb) + sb);
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
  chain_wait();
  chain_release();
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
    collide_rest<LAT, ODD>(L, C, x, y, z, m, uF, h, omega, cf, f[0]);
#pragma unroll
    for (int i = 1; i < Q; i += 2) collide_pair<LAT, ODD>(L, C, i, x, y, z, m, uF, h, omega, cf, f[i], f[i + 1]);
  }
  if (RED) block_reduce_store(acc, L.partials, blockIdx.x);
}

// Small lattices: four warps share the operations of 32 cells.  The FP64 pipe
// of an SM quarter takes 64 clocks for a warp instruction however few lanes
// are active, so 64 x 64 cells as 128 warps keep 128 of the 608 quarters busy
// for the 240 operations of a cell, one after another.  Here warp 0 sums M0,
// warps 1, 2 and 3 the momentum components (3 also the quadrature); after rho~,
// which all form, warp a takes F_a and u_a; then the opposite pairs are dealt
// to the warps.  About 95 operations deep for D2Q9; the same operations on
// every value, so the same bits.  Worth it while the chip is not full: up to
// two such blocks an SM, 9728 cells (make_launch_exact).  64 x 64 D2Q9: 6.1 us
// a step (9.0 with one warp for 32 cells).
constexpr int kSplit = 4;

template <class LAT, bool ODD>
__global__ void __launch_bounds__(32 * kSplit) step_exact_split_kernel(const LatticeDev *__restrict__ Lp, int k) {
  constexpr int Q = LAT::Q, D = LAT::D;
  __shared__ double sM[32], sI[32], sJ[3][32], sF[3][32], su[3][32];
  const LatticeDev &L = *Lp;
  const int lane = threadIdx.x, w = threadIdx.y;
  const long long idx = (long long)blockIdx.x * 32 + lane;
  const long long plane_cells = (long long)L.nx * L.ny;
  const bool inside = idx < plane_cells * L.nz;
  const int z = D == 3 ? (int)(idx / plane_cells) : 0;
  const long long rest = D == 3 ? idx - z * plane_cells : idx;
  const int y = D >= 2 ? (int)(rest / L.nx) : 0;
  const int x = (int)(rest - (long long)y * L.nx);
  const bool fluid = inside && !(L.walls && solid_at(L.walls, x, y, z, 0, 0, 0, L.nx, L.ny, L.nz));
  const long long n = L.n + k;
  const Coords C = fluid ? make_coords(x, y, z, L.nx, L.ny, L.nz, L.nxp) : make_coords(0, 0, 0, 1, 1, 1, 8);
  chain_wait();
  chain_release();
  double f[Q];
  MacroD m;
  if (fluid) {
    // every warp reads the cell's slots before the first barrier; they are
    // overwritten after it
    const double *pop = static_cast<const double *>(L.pop);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const SlotAddr a = slot_of<LAT>(L, C, ODD, i, x, y, z);
      f[i] = pop[(long long)a.slot * L.plane + a.cell];
    }
    if (w == 0) sM[lane] = sum_m0<LAT>(f);
    if (w == 1) sJ[0][lane] = sum_j<LAT>(f, 0);
    if (w == 2 && D >= 2) sJ[1][lane] = sum_j<LAT>(f, 1);
    if (w == 3) {
      if (D == 3) sJ[2][lane] = sum_j<LAT>(f, 2);
      double ep[3], em[3], ec;
      phi_stencil<LAT, true>(L, n, C, ec, ep, em);
      sI[lane] = quad_exact(L, ec, ep, em);
    }
  }
  __syncthreads();
  if (fluid) {
    m.M0 = sM[lane];
    m.rho = m.M0 / sI[lane];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      if (w != a) continue;
      double ep[3], em[3], ec;
      phi_stencil<LAT, true>(L, n, C, ec, ep, em);
      const double F = force_exact<true>(L, n, C, a, m.rho, ep[a], em[a]);
      sF[a][lane] = F;
      su[a][lane] = __fma_rn(0.5, F, sJ[a][lane]) / m.M0;
    }
  }
  __syncthreads();
  if (!fluid) return;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    m.F[a] = a < D ? sF[a][lane] : 0.0;
    m.u[a] = a < D ? su[a][lane] : 0.0;
  }
  const double usq = dot_d<LAT>(m.u, m.u), uF = dot_d<LAT>(m.u, m.F), h = 1.5 * usq;
  if (w == kSplit - 1) collide_rest<LAT, ODD>(L, C, x, y, z, m, uF, h, L.omega, L.cf, f[0]);
#pragma unroll
  for (int i = 1; i < Q; i += 2)
    if (w == (i / 2) % kSplit) collide_pair<LAT, ODD>(L, C, i, x, y, z, m, uF, h, L.omega, L.cf, f[i], f[i + 1]);
}

// ---- moments, initialisation, populations (FP64 arithmetic) -----------------

template <class LAT>
__global__ void moments_kernel(const LatticeDev *__restrict__ Lp, double *rho, double *p, double *u,
                               float *rho_f, float *p_f, float *u_f) {
  const LatticeDev &L = *Lp;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= L.nx || y >= L.ny) return;
  moments_cell<LAT>(L, x, y, z, rho, p, u, rho_f, p_f, u_f);
}

// Initial state of FP64 and FP16 lattices (FP32: fields_ff.cu).
template <class LAT, bool F64>
__global__ void init_kernel(const LatticeDev *__restrict__ Lp, const double *p0, const double *u0, int mode) {
  const LatticeDev &L = *Lp;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= L.nx || y >= L.ny) return;
  init_cell<LAT, F64>(L, x, y, z, p0, u0, mode);
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
  cudaError_t e;
  if (odd) {
    if (red) e = launch_chained(step_exact_kernel<LAT, true, true, EXT>, ls.grid, ls.block, 0, s, k > 0, L_dev, k);
    else e = launch_chained(step_exact_kernel<LAT, true, false, EXT>, ls.grid, ls.block, 0, s, k > 0, L_dev, k);
  } else {
    if (red) e = launch_chained(step_exact_kernel<LAT, false, true, EXT>, ls.grid, ls.block, 0, s, k > 0, L_dev, k);
    else e = launch_chained(step_exact_kernel<LAT, false, false, EXT>, ls.grid, ls.block, 0, s, k > 0, L_dev, k);
  }
  return e;
}

template <class LAT>
static cudaError_t launch_exact_lat(const LatticeDev *L_dev, bool ext, bool odd, int red, int k,
                                    const StepLaunch &ls, cudaStream_t s) {
  return ext ? launch_exact_ext<LAT, true>(L_dev, odd, red, k, ls, s)
             : launch_exact_ext<LAT, false>(L_dev, odd, red, k, ls, s);
}

template <class LAT>
static cudaError_t launch_exact_split(const LatticeDev *L_dev, bool odd, int k, const StepLaunch &ls, cudaStream_t s) {
  const dim3 block(32, kSplit);
  return odd ? launch_chained(step_exact_split_kernel<LAT, true>, ls.grid, block, 0, s, k > 0, L_dev, k)
             : launch_chained(step_exact_split_kernel<LAT, false>, ls.grid, block, 0, s, k > 0, L_dev, k);
}

cudaError_t launch_step_exact(const LatticeDev &h, const LatticeDev *L_dev, bool odd, int red, int k,
                              const StepLaunch &ls, cudaStream_t s) {
  const bool ext = h.drag_model || h.les;
  if (ls.exact_split && !ext && !red) {
    switch (h.lattice) {
      case 0: return launch_exact_split<D2Q9>(L_dev, odd, k, ls, s);
      case 1: return launch_exact_split<D3Q19>(L_dev, odd, k, ls, s);
      case 2: return launch_exact_split<D3Q27>(L_dev, odd, k, ls, s);
      case 3: return launch_exact_split<D1Q3>(L_dev, odd, k, ls, s);
    }
  }
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
  // single-precision outputs of a reduced-precision lattice: float-float
  if (h.storage != 0 && !rho && !p && !u) return launch_moments_ff(h, L_dev, rho_f, p_f, u_f, s);
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
  if (h.storage == 1) return launch_init_ff(h, L_dev, p0, u0, mode, s);
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
