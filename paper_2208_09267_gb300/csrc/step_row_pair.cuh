// step_row_pair.cuh -- the row kernel's per-cell update for two adjacent
// cells per lane, FP16-shifted storage, plain steps (no check sums).
//
// Each operation of update_row_chunk is applied to the cells x and x + 1 at
// once as a packed FP32 pair operation (fma/add/mul .rn.f32x2: per
// component the same IEEE operation with the same rounding as the scalar
// one); divisions and the stochastic rounding stay per cell, with the same
// random bits.  So every stored value is bit-identical to update_row_chunk's
// for the same cell.  What the pair saves is issue slots: one instruction
// for two cells' arithmetic, one 4-byte shared-memory access for the two
// cells' halves of an unshifted row, and the index arithmetic done once for
// both cells.  SR (stochastic rounding, else nearest) is a template argument
// and the quadrature axes enter as weights: with a branch per stored pair the
// compiler could not interleave the independent pairs.
#pragma once

#include <cuda_fp16.h>

namespace lbm {

typedef float2 P2;  // the values of cells x and x + 1
__device__ __forceinline__ float lo(P2 a) { return a.x; }
__device__ __forceinline__ float hi(P2 a) { return a.y; }
__device__ __forceinline__ P2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ P2 f2s(float a) { return make_float2(a, a); }
__device__ __forceinline__ P2 fma2(P2 a, P2 b, P2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ P2 add2(P2 a, P2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ P2 mul2(P2 a, P2 b) { return __fmul2_rn(a, b); }
// a - b, exactly as the scalar subtraction rounds it (b * -1 is exact)
__device__ __forceinline__ P2 sub2(P2 a, P2 b) { return fma2(b, f2s(-1.0f), a); }

__device__ __forceinline__ P2 neg2(P2 a) { return f2(-lo(a), -hi(a)); }

// two halves at an even index (one 4-byte load)
__device__ __forceinline__ P2 ld_h2(const __half *p) {
  return __half22float2(*reinterpret_cast<const __half2 *>(p));
}
// two floats at an even index (one 8-byte load)
__device__ __forceinline__ P2 ld_f2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ float ldh(const __half *p) { return __half2float(*p); }

// 1/b and a/b of both cells, rounded as the IEEE operators of the scalar
// update round them: Newton's iteration on the hardware's approximate
// reciprocal, then Markstein's correction q + y (a - b q) with the exact FMA
// remainder, applied until the remainder is that of the nearest quotient (IBM
// J. Res. Dev. 34, 1990).  Packed for two cells it takes a third of the
// instructions of four operator divisions and no branch.  Range: b between
// 2^-125 and 2^100 and a between 2^-98 and 2^61 in magnitude, so that no
// approximation is flushed and no remainder loses bits.  M0 is there, or zero
// (u is not finite either way), for the densities of packed_division_range: it
// is a float sum of multiples of 2^-98 (halves times 2^-24 or more times
// weights, and differences of halves times rho0).  int phi dV comes times
// kDivScale, a power of two that changes no rounding.
__device__ __forceinline__ float rcp_approx(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ P2 recip2(P2 b) {
  const P2 nb = neg2(b);
  P2 y = f2(rcp_approx(lo(b)), rcp_approx(hi(b)));
  y = fma2(y, fma2(nb, y, f2s(1.0f)), y);
  return fma2(y, fma2(nb, y, f2s(1.0f)), y);
}
__device__ __forceinline__ P2 quot2(P2 a, P2 b, P2 y) {
  const P2 nb = neg2(b);
  P2 q = mul2(a, y);
  q = fma2(fma2(nb, q, a), y, q);
  return fma2(fma2(nb, q, a), y, q);
}
// Store the low (hi = false) or high halves of the two cells' packed
// results: at the even index x (both cells, one 4-byte store) when the
// destinations are adjacent, else one by one (the second cell only if it
// exists).
__device__ __forceinline__ void st_h2(__half *row, unsigned ha, unsigned hb, bool high, bool adjacent, int xa,
                                      int da, int db, bool vb) {
  if (adjacent) {
    *reinterpret_cast<unsigned *>(row + xa) = __byte_perm(ha, hb, high ? 0x7632 : 0x5410);
  } else {
    row[da] = __ushort_as_half((unsigned short)(high ? ha >> 16 : ha & 0xffffu));
    if (vb) row[db] = __ushort_as_half((unsigned short)(high ? hb >> 16 : hb & 0xffffu));
  }
}

// RESHIFT: the step after a phi refresh (decode with the old shift, encode
// with the new one); as a one-cell update it took 0.45 ms of a refresh interval
// of ten 256^3 steps at 0.28.
// Update cells xa and xa + 1 (xa even) of one staged row.  A second cell
// past the end of the row (odd nx) repeats the first one's indices; its
// results are discarded (the adjacent stores write the row's padding slot).
template <class LAT, bool ODD, bool WALLS, int PITCH, bool INPLACE, bool SR, bool TILED = true, bool RESHIFT = false>
__device__ __forceinline__ void update_row_pair(const LatticeDev &L, unsigned char *stage, int t,
                                                const RowCtx &rc, long long n, float dn, float dn_force,
                                                int xa) {
  using Lay = RowLayout<LAT, __half, ODD, PITCH>;
  constexpr int Q = LAT::Q, D = LAT::D;
  const int nx = L.nx;
  if (xa >= nx) return;
  const int sp = TILED ? L.nxp : PITCH, tt = TILED ? t : 0;
  // row t of the staged tile (the layout of update_row_chunk)
  const __half *prow = reinterpret_cast<const __half *>(stage) + tt * sp;
  const __half *srow = reinterpret_cast<const __half *>(stage + Lay::kSigOff) + (ODD ? tt + 1 : tt) * sp;
  const float *e0p = reinterpret_cast<const float *>(stage + Lay::kEpsOff) + (tt + 1) * sp;
  const float *ezm = reinterpret_cast<const float *>(stage + Lay::kEpsOff) + 3 * PITCH + tt * sp;
  const float *d0p = reinterpret_cast<const float *>(stage + Lay::kDepsOff) + (tt + 1) * sp;
  const float *dzm = reinterpret_cast<const float *>(stage + Lay::kDepsOff) + 3 * PITCH + tt * sp;
  const bool tv = L.has_deps != 0;
  const float rho0 = L.rho0f;
  const float inv_scale = L.inv_scale, scale = L.scale;
  __half *__restrict__ pop = static_cast<__half *>(L.pop);
  const long long plane = L.plane;
  const float omega = L.omegaf;
  const float om1 = 1.0f - omega;
  const float cf3 = L.cf3f, cf9 = L.cf9f;
  const unsigned qa = L.quad_axes;
  const bool vb = xa + 1 < nx;
  const int xb = vb ? xa + 1 : xa;
  const int xsa[3] = {xa == 0 ? nx - 1 : xa - 1, xa, xa == nx - 1 ? 0 : xa + 1};
  const int xsb[3] = {xb == 0 ? nx - 1 : xb - 1, xb, xb == nx - 1 ? 0 : xb + 1};
  const int cell = rc.base[1][1] + xa;

#define EPS_ROW(dy, dz) ((dz) == 0 ? e0p + (dy) * sp : ((dz) < 0 ? ezm : ezm + PITCH))
#define DEPS_ROW(dy, dz) ((dz) == 0 ? d0p + (dy) * sp : ((dz) < 0 ? dzm : dzm + PITCH))
#define SIG_ROW(dy, dz) (ODD ? srow + sig_block<LAT>(dz) * 3 * PITCH + (dy) * sp : srow)
  // a half row at the two cells' positions shifted by s in x (s = 0: the
  // cells themselves, one aligned load)
#define LD_H_SHIFT(row, s) ((s) == 0 ? ld_h2((row) + xa) : f2(ldh((row) + xsa[1 + (s)]), ldh((row) + xsb[1 + (s)])))
#define OWN_SRC(i) (!ODD || (i) == 0 || (WALLS && ((rc.solid >> ((1 - LAT::c((i), 2)) * 3 + (1 - LAT::c((i), 1)))) & 1u)))
#define OWN_DST(i) (!ODD || (i) == 0 || (WALLS && ((rc.solid >> ((1 + LAT::c((i), 2)) * 3 + (1 + LAT::c((i), 1)))) & 1u)))

  const P2 sig_own = ld_h2(SIG_ROW(0, 0) + xa);
  const __half *__restrict__ srd = L.sig_rd;
  const P2 s_x = mul2(f2s(rho0), RESHIFT ? ld_h2(srd + cell) : sig_own);
  const P2 ms_x = f2(-lo(s_x), -hi(s_x));
  const P2 rho2 = f2s(rho0), scale2 = f2s(scale);

  // 1. decode (update_row_chunk step 1, in storage units)
  P2 d[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int cx = LAT::c(i, 0), cy = LAT::c(i, 1), cz = LAT::c(i, 2);
    const __half *pr = prow + i * PITCH;
    if (OWN_SRC(i)) {
      d[i] = ld_h2(pr + xa);
    } else {
      const P2 q = LD_H_SHIFT(pr, -cx);
      const P2 sw = RESHIFT ? LD_H_SHIFT(srd + rc.base[1 - cz][1 - cy], -cx) : LD_H_SHIFT(SIG_ROW(-cy, -cz), -cx);
      d[i] = fma2(fma2(rho2, sw, ms_x), scale2, q);
    }
  }

  // 2. moments (the storage scale 2^-k folded into the weights: exact)
  P2 dM, j0, j1, j2 = f2s(0.f);
  {
    const float is = inv_scale;
    dM = mul2(f2s((float)LAT::w(0) * is), d[0]);
    bool f0 = true, f1 = true, f2_ = true;
#pragma unroll
    for (int i = 1; i < Q; ++i) {
      const float w = (float)LAT::w(i) * is;
      const P2 wp = f2s(w), wm = f2s(-w);
      dM = fma2(wp, d[i], dM);
#define ADD_J(J, FIRST, A)                                        \
  if (LAT::c(i, A) != 0) {                                        \
    const P2 ws = LAT::c(i, A) > 0 ? wp : wm;                     \
    J = FIRST ? mul2(ws, d[i]) : fma2(ws, d[i], J);               \
    FIRST = false;                                                \
  }
      ADD_J(j0, f0, 0)
      ADD_J(j1, f1, 1)
      if (D == 3) { ADD_J(j2, f2_, 2) }
#undef ADD_J
    }
  }
  const P2 M0 = add2(s_x, dM);

  // 3. phi at time n on the stencil (x - 1 of the second cell is the first
  //    cell; x + 1 of the first is the second, unless the first is the
  //    row's last cell)
  const float *e0r = EPS_ROW(0, 0);
  P2 e_c = ld_f2(e0r + xa);
  P2 e_xm = f2(e0r[xsa[0]], lo(e_c)), e_xp = f2(vb ? hi(e_c) : e0r[xsa[2]], e0r[xsb[2]]);
  P2 e_yp = ld_f2(EPS_ROW(1, 0) + xa), e_ym = ld_f2(EPS_ROW(-1, 0) + xa);
  P2 e_zp = e_c, e_zm = e_c;
  if (D == 3) {
    e_zp = ld_f2(EPS_ROW(0, 1) + xa);
    e_zm = ld_f2(EPS_ROW(0, -1) + xa);
  }
  if (tv) {
    const P2 dn2 = f2s(dn);
    const float *d0r = DEPS_ROW(0, 0);
    const P2 t_c = ld_f2(d0r + xa);
    e_c = fma2(dn2, t_c, e_c);
    e_xp = fma2(dn2, f2(vb ? hi(t_c) : d0r[xsa[2]], d0r[xsb[2]]), e_xp);
    e_xm = fma2(dn2, f2(d0r[xsa[0]], lo(t_c)), e_xm);
    e_yp = fma2(dn2, ld_f2(DEPS_ROW(1, 0) + xa), e_yp);
    e_ym = fma2(dn2, ld_f2(DEPS_ROW(-1, 0) + xa), e_ym);
    if (D == 3) {
      e_zp = fma2(dn2, ld_f2(DEPS_ROW(0, 1) + xa), e_zp);
      e_zm = fma2(dn2, ld_f2(DEPS_ROW(0, -1) + xa), e_zm);
    }
  }

  // 4.-6. quadrature, density, forces, velocity
  // (an axis outside eq. (quad) enters with weight 0: no branch)
  P2 nb = mul2(f2s(qa & 1u ? 1.f : 0.f), add2(e_xp, e_xm));
  nb = fma2(f2s(qa & 2u ? 1.f : 0.f), add2(e_yp, e_ym), nb);
  if (D == 3) nb = fma2(f2s(qa & 4u ? 1.f : 0.f), add2(e_zp, e_zm), nb);
  const P2 I = fma2(f2s(L.qw0f), e_c, mul2(f2s(L.qw1f), nb));  // kDivScale int phi dV
  const P2 invM = recip2(M0);
  const P2 rho = quot2(M0, I, recip2(I));  // rho~ / kDivScale
  const P2 pc2 = mul2(rho, f2s(0.5f / 3.0f * kDivScale));
  P2 F0 = fma2(pc2, sub2(e_xp, e_xm), f2s(L.gf[0]));
  P2 F1 = fma2(pc2, sub2(e_yp, e_ym), f2s(L.gf[1]));
  P2 F2 = D == 3 ? fma2(pc2, sub2(e_zp, e_zm), f2s(L.gf[2])) : f2s(0.f);
  if (L.has_force) {
    const float *__restrict__ fo = static_cast<const float *>(L.force);
    const long long N = L.ncell;
    P2 a0 = ld_f2(fo + cell), a1 = ld_f2(fo + N + cell);
    P2 a2 = D == 3 ? ld_f2(fo + 2 * N + cell) : f2s(0.f);
    if (L.has_dforce) {
      const float *__restrict__ df = static_cast<const float *>(L.dforce);
      const P2 dnf = f2s(dn_force);
      a0 = fma2(dnf, ld_f2(df + cell), a0);
      a1 = fma2(dnf, ld_f2(df + N + cell), a1);
      if (D == 3) a2 = fma2(dnf, ld_f2(df + 2 * N + cell), a2);
    }
    F0 = add2(F0, a0);
    F1 = add2(F1, a1);
    F2 = add2(F2, a2);
  }
  const P2 half2c = f2s(0.5f);
  const P2 u0 = mul2(fma2(half2c, F0, j0), invM);
  const P2 u1 = mul2(fma2(half2c, F1, j1), invM);
  const P2 u2 = D == 3 ? mul2(fma2(half2c, F2, j2), invM) : f2s(0.f);
  const P2 usq = fma2(u0, u0, fma2(u1, u1, mul2(u2, u2)));
  const P2 uF = fma2(u0, F0, fma2(u1, F1, mul2(u2, F2)));

  // 7.-8. collide and stream (update_row_chunk's FP16 branch)
  const P2 m15usq = mul2(f2s(-1.5f), usq);
  const float sc = scale;
  const float omega_s = omega * sc, cf3_s = cf3 * sc, cf9_s = cf9 * sc;
  const P2 m3uF_s = mul2(f2s(-cf3 * sc), uF);
  SRng rng_a((unsigned)cell, n), rng_b((unsigned)(cell + 1), n);
  const P2 om1_2 = f2s(om1), sc2 = f2s(sc), msc2 = f2s(-sc);
  __half *orow = INPLACE ? reinterpret_cast<__half *>(stage) + tt * sp : nullptr;

  // destination row of population i: the staged block that f_opp(i) came
  // from, or the population plane (own slot: plane opp(i) of this row; else plane i of
  // row (y + c_iy, z + c_iz))
  const P2 enc_own = RESHIFT ? fma2(f2s(-rho0), sig_own, s_x) : f2s(0.f);
#define DST_ROW(i, own)                                                                              \
  ((INPLACE) ? orow + opp_of(i) * PITCH                                                              \
          : ((own) ? pop + opp_of(i) * plane + rc.base[1][1]                                         \
                   : pop + (i) * plane + rc.base[1 + LAT::c((i), 2)][1 + LAT::c((i), 1)]))

  {
    // rest population
    P2 v = fma2(om1_2, d[0], fma2(f2s(omega_s), fma2(M0, m15usq, dM), m3uF_s));
    if (RESHIFT) v = fma2(enc_own, sc2, v);
    __half ha, hb;
    if (SR) {
      ha = half_sr(lo(v), rng_a.next13());
      hb = half_sr(hi(v), rng_b.next13());
    } else {
      ha = __float2half_rn(lo(v));
      hb = __float2half_rn(hi(v));
    }
    __half *row = DST_ROW(0, true);
    *reinterpret_cast<__half2 *>(row + xa) = __halves2half2(ha, hb);
  }
  const P2 oM03 = mul2(f2s(3.0f * omega_s), M0);
#pragma unroll
  for (int i = 1; i < Q; i += 2) {
    const int cx = LAT::c(i, 0), cy = LAT::c(i, 1), cz = LAT::c(i, 2);
    P2 cu = f2s(0.f), cF = f2s(0.f);
    bool any = false;
#define ADD_C(A, UA, FA)                                                   \
  if (LAT::c(i, A) != 0) {                                                 \
    if (LAT::c(i, A) > 0) {                                                \
      cu = any ? add2(cu, UA) : UA;                                        \
      cF = any ? add2(cF, FA) : FA;                                        \
    } else {                                                               \
      cu = any ? sub2(cu, UA) : neg2(UA);                                  \
      cF = any ? sub2(cF, FA) : neg2(FA);                                  \
    }                                                                      \
    any = true;                                                            \
  }
    ADD_C(0, u0, F0)
    ADD_C(1, u1, F1)
    ADD_C(2, u2, F2)
#undef ADD_C
    const P2 t = fma2(M0, fma2(mul2(f2s(4.5f), cu), cu, m15usq), dM);
    const P2 A = fma2(f2s(omega_s), t, fma2(mul2(f2s(cf9_s), cu), cF, m3uF_s));
    const P2 B = fma2(oM03, cu, mul2(f2s(cf3_s), cF));
    P2 va = fma2(om1_2, d[i], add2(A, B));
    P2 vb2 = fma2(om1_2, d[i + 1], sub2(A, B));
    // encode against the shift of the storage cell (update_row_chunk's
    // ENCODE_POP).  The shift differences are formed again, not kept from the
    // decode: 36 registers against a load and two conversions each, and 96
    // registers a thread give a third more warps.
    const bool own_a = OWN_DST(i), own_b = OWN_DST(i + 1);
    if (RESHIFT && own_a) va = fma2(enc_own, sc2, va);
    if (RESHIFT && own_b) vb2 = fma2(enc_own, sc2, vb2);
    if (!own_a) {
      if (!RESHIFT && !OWN_SRC(i + 1))
        va = fma2(fma2(rho2, LD_H_SHIFT(SIG_ROW(cy, cz), cx), ms_x), msc2, va);
      else
        va = fma2(fma2(f2s(-rho0), LD_H_SHIFT(SIG_ROW(cy, cz), cx), s_x), sc2, va);
    }
    if (!own_b) {
      if (!RESHIFT && !OWN_SRC(i))
        vb2 = fma2(fma2(rho2, LD_H_SHIFT(SIG_ROW(-cy, -cz), -cx), ms_x), msc2, vb2);
      else
        vb2 = fma2(fma2(f2s(-rho0), LD_H_SHIFT(SIG_ROW(-cy, -cz), -cx), s_x), sc2, vb2);
    }
    unsigned ha, hb;  // (population i, population i + 1) of each cell
    if (SR) {
      ha = half2_sr(lo(va), lo(vb2), rng_a.next32());
      hb = half2_sr(hi(va), hi(vb2), rng_b.next32());
    } else {
      ha = (unsigned)__half_as_ushort(__float2half_rn(lo(va))) | ((unsigned)__half_as_ushort(__float2half_rn(lo(vb2))) << 16);
      hb = (unsigned)__half_as_ushort(__float2half_rn(hi(va))) | ((unsigned)__half_as_ushort(__float2half_rn(hi(vb2))) << 16);
    }
    // population i goes to x + c_ix unless it stays; i + 1 to x - c_ix
    st_h2(DST_ROW(i, own_a), ha, hb, false, own_a || cx == 0, xa, own_a ? xa : xsa[1 + cx],
          own_a ? xb : xsb[1 + cx], vb);
    st_h2(DST_ROW(i + 1, own_b), ha, hb, true, own_b || cx == 0, xa, own_b ? xa : xsa[1 - cx],
          own_b ? xb : xsb[1 - cx], vb);
  }
#undef DST_ROW
#undef EPS_ROW
#undef DEPS_ROW
#undef SIG_ROW
#undef LD_H_SHIFT
#undef OWN_SRC
#undef OWN_DST
}

}  // namespace lbm
