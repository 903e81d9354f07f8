// fields_ff.cu -- single-precision moments of FP32 and FP16 lattices and the
// initial state of FP32 lattices, in float-float arithmetic (ff.cuh).
//
// Both were FP64 kernels and bound by the FP64 pipe (2 lanes per clock and
// SM): 465 FP64 operations per D3Q27 cell took 27 ms on 512 x 256 x 256 cells,
// where the memory traffic takes under a millisecond.  The stored values are floats or
// halves, so a pair of floats holds every intermediate to 48 bits, enough
// that the single-precision results round as the FP64 ones do (values that
// cancel, p and u near zero, to about 1e-14 absolute).  Now 2.2 ms on those
// cells at an even time (half of the measured copy bandwidth; FP32 arithmetic
// bounds it) and 7.6 ms at an odd one, where every value carries its slot's
// shift; 0.96 and 2.9 ms on D3Q19 256^3 FP16.  An FP32 initial state from rest
// takes 3.3 ms on the same D3Q27 cells (before 29).  Moments in double precision (rho, p, u as
// double) keep the FP64 kernel.
#include "exact.cuh"
#include "ff.cuh"

namespace lbm {

// Cells with infinities, NaN or values beyond the float range: the FP64
// arithmetic of exact.cuh, so that such states read back as they always did.
template <class LAT>
__device__ __noinline__ void moments_cell_wide(const LatticeDev *L, int x, int y, int z, float *rho, float *p,
                                               float *u) {
  moments_cell<LAT>(*L, x, y, z, nullptr, nullptr, nullptr, rho, p, u);
}

template <class LAT>
__device__ __noinline__ void init_cell_wide(const LatticeDev *L, int x, int y, int z, const double *p0,
                                            const double *u0, int mode) {
  init_cell<LAT, false>(*L, x, y, z, p0, u0, mode);
}

// The descriptor's doubles as float-float, converted once per block.
struct FieldConsts {
  ff rho0, qw0, qw1, g[3], drag_lin, drag_q, dn, dnf;
};

__device__ __forceinline__ void load_consts(const LatticeDev &L, FieldConsts &k) {
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    k.rho0 = ff_of(L.rho0);
    k.qw0 = ff_of(L.qw0);
    k.qw1 = ff_of(L.qw1);
    for (int a = 0; a < 3; ++a) k.g[a] = ff_of(L.g[a]);
    k.dn = ff_of((double)(L.n - L.n_eps));
    k.dnf = ff_of((double)(L.n - L.n_force));
    if (L.drag_model) {
      k.drag_lin = ff_of(L.drag_c1 * ((L.tau0 - 0.5) / 3.0) / (L.drag_d * L.drag_d));
      k.drag_q = ff_of(L.drag_c2 / L.drag_d);
    }
  }
  __syncthreads();
}

__device__ __forceinline__ ff field_at(const void *f, const void *df, bool tv, long long m, ff dn) {
  const ff e = ff_of(__ldg(static_cast<const float *>(f) + m));
  return tv ? dn * __ldg(static_cast<const float *>(df) + m) + e : e;
}

template <class LAT>
__device__ __forceinline__ ff weight(int i) {
  const double w = LAT::w(i);
  return {(float)w, (float)(w - (double)(float)w)};
}

struct MacroF {
  ff rho, u[3], F[3];
};

// phi on the face stencil, int phi dV of eq. (quad), and from M0 and J the
// density, force and velocity (step_exact.cu's macro_from_sums).
template <class LAT>
__device__ __forceinline__ void macro_ff(const LatticeDev &L, const FieldConsts &k, const Coords &C, ff M0,
                                         const ff *J, MacroF &m) {
  constexpr int D = LAT::D;
  const bool tv = L.has_deps != 0;
  const ff e_c = field_at(L.eps, L.deps, tv, C.at(0, 0, 0), k.dn);
  ff diff[3], nb = ff_of(0.f);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const ff ep = field_at(L.eps, L.deps, tv, C.at(a == 0, a == 1, a == 2), k.dn);
    const ff em = field_at(L.eps, L.deps, tv, C.at(-(a == 0), -(a == 1), -(a == 2)), k.dn);
    diff[a] = ep - em;
    if (L.quad_axes & (1u << a)) nb = nb + (ep + em);
  }
  const ff I = k.qw0 * e_c + k.qw1 * nb;
  m.rho = M0 / I;
  const ff third = ff_of(1.0 / 3.0);
  const ff hpc = scaled(m.rho * third, 0.5f);
  const long long cell = C.at(0, 0, 0);
  ff b[3];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    m.F[a] = k.g[a] + hpc * diff[a];
    if (L.has_force) {
      const long long off = (long long)a * L.ncell;
      m.F[a] = m.F[a] + field_at(static_cast<const float *>(L.force) + off,
                                 static_cast<const float *>(L.dforce) + off, L.has_dforce != 0, cell, k.dnf);
    }
    b[a] = J[a] + scaled(m.F[a], 0.5f);
  }
  ff den = M0;
  if (L.drag_model) {
    // the drag law, implicit in eq. (velocity): see macro_from_sums
    const ff one_m = ff_of(1.f) - e_c;
    const ff lin = m.rho * k.drag_lin * one_m * one_m / e_c;
    const ff bq = m.rho * k.drag_q * one_m;
    ff bb = b[0] * b[0];
#pragma unroll
    for (int a = 1; a < D; ++a) bb = bb + b[a] * b[a];
    const ff bn = ff_sqrt(bb);
    const ff A = M0 + scaled(lin, 0.5f);
    const ff sp = scaled(bn, 2.0f) / (A + ff_sqrt(A * A + scaled(bq * bn, 2.0f)));
    den = A + scaled(bq * sp, 0.5f);
    const ff beta = lin + bq * sp;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      m.u[a] = b[a] / den;
      m.F[a] = m.F[a] - beta * m.u[a];
    }
    return;
  }
#pragma unroll
  for (int a = 0; a < D; ++a) m.u[a] = b[a] / den;
}

// Moments of one cell.  Sums run over opposite pairs: their sum
// enters M0, their difference J, by weight class (at most four).  The cell's
// own rest state rho0 sigma(x) is left out of the sums (the weights add to
// one, the velocities to zero) and added to M0; at even n (ODD = false) all
// values are stored against it and the sums are over the stored values alone.
template <class LAT, class ST, bool ODD>
__device__ __forceinline__ void moments_cell_ff(const LatticeDev *__restrict__ Lp, const FieldConsts &k, int x, int y,
                                                int z, float *rho, float *p, float *u) {
  constexpr int Q = LAT::Q, D = LAT::D;
  const LatticeDev &L = *Lp;
  const Coords C = make_coords(x, y, z, L.nx, L.ny, L.nz, L.nxp);
  // outputs are dense: index (z*ny + y)*nx + x, N = nx*ny*nz
  const long long o = ((long long)z * L.ny + y) * L.nx + x;
  const long long N = (long long)L.nx * L.ny * L.nz;
  if (L.walls && solid_at(L.walls, x, y, z, 0, 0, 0, L.nx, L.ny, L.nz)) {
    if (rho) rho[o] = 0.f;
    if (p) p[o] = 0.f;
    if (u)
      for (int a = 0; a < 3; ++a) u[a * N + o] = 0.f;
    return;
  }
  const long long cell = C.at(0, 0, 0);
  const ST *pop = static_cast<const ST *>(L.pop);
  const float s0 = __half2float(L.sig_rd[cell]), inv_scale = L.inv_scale;
  // stored values (times 2^-k: exact) and, at odd n, the differences of the
  // slots' shifts from the cell's own (exact)
  float q[Q], ds[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const SlotAddr a = slot_of<LAT>(L, C, ODD, i, x, y, z);
    q[i] = PopIO<ST>::ld(pop + (long long)a.slot * L.plane + a.cell) * inv_scale;
    ds[i] = ODD && i != 0 ? __half2float(L.sig_rd[a.cell]) - s0 : 0.f;
  }
  auto value = [&](int i) -> ff { return ODD ? k.rho0 * ds[i] + q[i] : ff_of(q[i]); };
  ff M0 = k.rho0 * s0 + weight<LAT>(0) * q[0], J[3] = {ff_of(0.f), ff_of(0.f), ff_of(0.f)};
  // directions of one weight are consecutive: [1, 2D], edges, corners
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int first = c == 0 ? 1 : (c == 1 ? 2 * D + 1 : 19);
    const int last = c == 0 ? 2 * D : (c == 1 ? (Q < 19 ? Q - 1 : 18) : Q - 1);
    if (first > last) continue;
    ff_sum sM, sJ[3];
#pragma unroll
    for (int i = first; i <= last; i += 2) {
      const ff va = value(i), vb = value(i + 1);
      ff t = two_sum(va.h, vb.h), d = two_sum(va.h, -vb.h);
      if (ODD) {
        t.l = __fadd_rn(t.l, __fadd_rn(va.l, vb.l));
        d.l = __fadd_rn(d.l, __fsub_rn(va.l, vb.l));
      }
      sM.add(t);
#pragma unroll
      for (int a = 0; a < D; ++a)
        if (LAT::c(i, a) != 0) sJ[a].add(LAT::c(i, a) > 0 ? d : -d);
    }
    const ff w = weight<LAT>(first);
    M0 = M0 + w * sM.total();
#pragma unroll
    for (int a = 0; a < D; ++a) J[a] = J[a] + w * sJ[a].total();
  }
  MacroF m;
  macro_ff<LAT>(L, k, C, M0, J, m);
  float sum = m.rho.h;
#pragma unroll
  for (int a = 0; a < D; ++a) sum += fabsf(m.u[a].h);
  if (!isfinite(sum)) {
    moments_cell_wide<LAT>(Lp, x, y, z, rho, p, u);
    return;
  }
  if (rho) rho[o] = m.rho.h;
  if (p) p[o] = ((m.rho - k.rho0) * ff_of(1.0 / 3.0)).h;
  if (u)
    for (int a = 0; a < 3; ++a) u[a * N + o] = a < D ? m.u[a].h : 0.f;
}

// At the device-side time: a captured call gives the fields of its replay, so
// the layout of the populations follows the descriptor's time, not the host's.
template <class LAT, class ST>
__global__ void __launch_bounds__(256) moments_ff_kernel(const LatticeDev *__restrict__ Lp, float *rho, float *p,
                                                         float *u) {
  const LatticeDev &L = *Lp;
  __shared__ FieldConsts k;
  load_consts(L, k);
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= L.nx || y >= L.ny) return;
  if (L.n & 1) moments_cell_ff<LAT, ST, true>(Lp, k, x, y, z, rho, p, u);
  else moments_cell_ff<LAT, ST, false>(Lp, k, x, y, z, rho, p, u);
}

// Write f_i/w_i = v to a slot: v - rho0 sigma against the newest shift.
__device__ __forceinline__ void store_ff(const LatticeDev &L, ff rho0, const SlotAddr &a, ff v) {
  static_cast<float *>(L.pop)[(long long)a.slot * L.plane + a.cell] = (v - rho0 * __half2float(L.sig_wr[a.cell])).h;
}

// FP32 storage.  (FP16 keeps the FP64 kernel: its stochastic rounding turns
// any difference in a stored half into another realisation of the noise.)
template <class LAT>
__global__ void __launch_bounds__(256) init_ff_kernel(const LatticeDev *__restrict__ Lp, const double *p0,
                                                      const double *u0, int mode) {
  constexpr int Q = LAT::Q, D = LAT::D;
  const LatticeDev &L = *Lp;
  __shared__ FieldConsts k;
  load_consts(L, k);
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z;
  if (x >= L.nx || y >= L.ny) return;
  if (L.walls && solid_at(L.walls, x, y, z, 0, 0, 0, L.nx, L.ny, L.nz)) return;
  const Coords C = make_coords(x, y, z, L.nx, L.ny, L.nz, L.nxp);
  // p0, u0 are dense arrays: index (z*ny + y)*nx + x, N = nx*ny*nz
  const long long kd = ((long long)z * L.ny + y) * L.nx + x;
  const long long N = (long long)L.nx * L.ny * L.nz;
  const bool odd = (L.n & 1) != 0, tv = L.has_deps != 0;
  ff u[3] = {ff_of(0.f), ff_of(0.f), ff_of(0.f)};
  if (u0)
    for (int a = 0; a < D; ++a) u[a] = ff_of(u0[a * N + kd]);
  ff mass = field_at(L.eps, L.deps, tv, C.at(0, 0, 0), k.dn);
  if (mode & 1) {
    ff nb = ff_of(0.f);
#pragma unroll
    for (int a = 0; a < D; ++a)
      if (L.quad_axes & (1u << a))
        nb = nb + (field_at(L.eps, L.deps, tv, C.at(a == 0, a == 1, a == 2), k.dn) +
                   field_at(L.eps, L.deps, tv, C.at(-(a == 0), -(a == 1), -(a == 2)), k.dn));
    mass = k.qw0 * mass + k.qw1 * nb;
  }
  const ff rt = p0 ? k.rho0 + ff_of(p0[kd]) * 3.0f : k.rho0;
  mass = rt * mass;
  if (mode & 2) {
    // the equilibrium's moments: M0 = mass, J = mass u
    ff J[3];
    for (int a = 0; a < D; ++a) J[a] = mass * u[a];
    MacroF m;
    macro_ff<LAT>(L, k, C, mass, J, m);
    for (int a = 0; a < D; ++a) u[a] = u[a] - scaled(m.F[a], 0.5f) / mass;
  }
  ff usq = u[0] * u[0];
#pragma unroll
  for (int a = 1; a < D; ++a) usq = usq + u[a] * u[a];
  const ff rest = ff_of(1.f) - usq * 1.5f;
  if (!isfinite(mass.h * rest.h * 1e6f)) {
    init_cell_wide<LAT>(Lp, x, y, z, p0, u0, mode);
    return;
  }
  store_ff(L, k.rho0, slot_of<LAT>(L, C, odd, 0, x, y, z), mass * rest);
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    ff cu = ff_of(0.f);
#pragma unroll
    for (int a = 0; a < D; ++a)
      if (LAT::c(i, a) != 0) cu = cu + (LAT::c(i, a) > 0 ? u[a] : -u[a]);
    const ff even = rest + cu * cu * 4.5f, lin = cu * 3.0f;
    store_ff(L, k.rho0, slot_of<LAT>(L, C, odd, i, x, y, z), mass * (even + lin));
    store_ff(L, k.rho0, slot_of<LAT>(L, C, odd, i + 1, x, y, z), mass * (even - lin));
  }
}

template <class LAT>
static void moments_lat(const LatticeDev &h, const LatticeDev *L_dev, float *rho, float *p, float *u,
                        const StepLaunch &ls, cudaStream_t s) {
  if (h.storage == 1) moments_ff_kernel<LAT, float><<<ls.grid, ls.block, 0, s>>>(L_dev, rho, p, u);
  else moments_ff_kernel<LAT, __half><<<ls.grid, ls.block, 0, s>>>(L_dev, rho, p, u);
}

cudaError_t launch_moments_ff(const LatticeDev &h, const LatticeDev *L_dev, float *rho, float *p, float *u,
                              cudaStream_t s) {
  const StepLaunch ls = make_launch(h.nx, h.ny, h.nz, 0, 0);
  switch (h.lattice) {
    case 0: moments_lat<D2Q9>(h, L_dev, rho, p, u, ls, s); break;
    case 1: moments_lat<D3Q19>(h, L_dev, rho, p, u, ls, s); break;
    case 2: moments_lat<D3Q27>(h, L_dev, rho, p, u, ls, s); break;
    case 3: moments_lat<D1Q3>(h, L_dev, rho, p, u, ls, s); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_init_ff(const LatticeDev &h, const LatticeDev *L_dev, const double *p0, const double *u0, int mode,
                           cudaStream_t s) {
  const StepLaunch ls = make_launch(h.nx, h.ny, h.nz, 0, 0);
  switch (h.lattice) {
    case 0: init_ff_kernel<D2Q9><<<ls.grid, ls.block, 0, s>>>(L_dev, p0, u0, mode); break;
    case 1: init_ff_kernel<D3Q19><<<ls.grid, ls.block, 0, s>>>(L_dev, p0, u0, mode); break;
    case 2: init_ff_kernel<D3Q27><<<ls.grid, ls.block, 0, s>>>(L_dev, p0, u0, mode); break;
    case 3: init_ff_kernel<D1Q3><<<ls.grid, ls.block, 0, s>>>(L_dev, p0, u0, mode); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace lbm
