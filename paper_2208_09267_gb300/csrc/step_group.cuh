// step_group.cuh -- the row-staged step of FP16 lattices: consumer groups and
// write-back in place.
//
// The tiles, their stage layout and the per-cell update are those of
// step_row.cuh.  What differs is how the warps are used, because FP16 moves
// half the bytes of FP32 for the same arithmetic and its consumer warps, not
// the memory, bound the step:
//
// * One block per SM: 16 consumer warps, two producers, two storers (96
//   registers a thread; each half of them with its own stages).  A tile
//   belongs to one group of PITCH/64 consumer warps (tile j to group j mod
//   NG), each warp updating 64 consecutive stored cells of it, two per lane.
//   A warp then waits for, and releases, only the tiles it works on: with
//   every warp dealt chunks of every tile, a quarter of all instructions went
//   into waiting for tiles.  The 64 cells run on over the rows of a tile, so
//   short rows leave no lanes idle.
// * The results overwrite the staged populations.  In the AA pattern a cell
//   writes exactly the slots it reads (f*_i goes where f_opp(i) came from), so
//   a staged block, once updated, is stored back to the rows it was loaded
//   from; no output stage is needed and the shared memory it took holds further
//   input stages instead.
//
// 256^3 D3Q19 with d_t phi: 287 us a step, 58.5 GLUPS, 0.72 of the measured
// copy bandwidth (381 us as two blocks of 6 consumers and output stages);
// 128^3: 42 us (56); D3Q27 512 x 256 x 256 with walls: 0.84 ms, 0.66 (0.98).
// The issue slots are 65-69 % used; what bounds it now is the instructions of
// the update (730 / 1054 per 64 cells, even / odd step).  One producer and one
// storer: 373 us at 256^3 (the groups wait for tiles).
#pragma once

#include "step_row.cuh"

namespace lbm {

constexpr int kGroupConsumers = 16;                         // consumer warps of a block
constexpr int kGroupHelpers = 2;                            // producers, and as many storers
constexpr int kGroupThreads = (kGroupConsumers + 2 * kGroupHelpers) * 32;

template <class LAT, int P>
struct GroupCfg {
  static constexpr int kGW = P / 64;                 // warps of a group: 64 cells each
  static constexpr int kNG = kGroupConsumers / kGW;  // groups
  static constexpr int kIn = RowLayout<LAT, __half, true, P>::kStageBytes;
  static constexpr int kInS = RowLayout<LAT, __half, true, P>::kDepsOff;  // static phi: no d_t phi blocks
  static constexpr int kBudget = (P == 512 ? 224 : 221) * 1024;  // of 227 KB; beside it the contexts
  static constexpr int kMax = 12;
  // a multiple of the helpers: a stage then belongs to one producer, one
  // storer and their groups, which run independently of the other half
  static constexpr int even(int n) { return n / kGroupHelpers * kGroupHelpers; }
  static constexpr int kNS = even(kBudget / kIn < kMax ? kBudget / kIn : kMax);
  static constexpr int kNSS = even(kBudget / kInS < kMax ? kBudget / kInS : kMax);
  static constexpr int kSmem = kNS * kIn > kNSS * kInS ? kNS * kIn : kNSS * kInS;
  static_assert(kNS >= kNG && kNG % kGroupHelpers == 0, "every group needs a stage");
};

// RED: a check step (one cell per lane), RS = 1: the step after a phi refresh.
template <class LAT, bool ODD, bool RED, bool WALLS, int PITCH, int RS, bool TILED>
__global__ void __launch_bounds__(kGroupThreads, 1)
    step_group_kernel(const LatticeDev *__restrict__ Lp, int k, int lay_static) {
  using Lay = RowLayout<LAT, __half, ODD, PITCH>;
  using Cfg = GroupCfg<LAT, PITCH>;
  constexpr int kMaxStage = Cfg::kNSS;
  constexpr bool kPair = !RED;
  const int NSTAGE = lay_static ? Cfg::kNSS : Cfg::kNS;
  const int kInStride = lay_static ? Lay::kDepsOff : Lay::kStageBytes;
  __shared__ LatticeDev Ls;
  __shared__ alignas(8) unsigned long long full[kMaxStage];   // the tile's copies have landed
  __shared__ alignas(8) unsigned long long done[kMaxStage];   // its group has updated it
  __shared__ alignas(8) unsigned long long empty[kMaxStage];  // its write-back has read the stage
  __shared__ RowCtx ctx[kMaxStage][TILED ? kMaxTileRows : 1];
  __shared__ int tile_nr[kMaxStage];
  // tiles issued by each producer: a parity wait tells a phase from the one
  // before it only, so a group waits for its tile's copies after they have
  // been issued (the stage's earlier tile is then through)
  __shared__ int issued[kGroupHelpers];
  __shared__ volatile int abort_flag;
  extern __shared__ __align__(128) unsigned char stages[];
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  {
    const int *src = reinterpret_cast<const int *>(Lp);
    int *dst = reinterpret_cast<int *>(&Ls);
    for (int w = tid; w < (int)(sizeof(LatticeDev) / sizeof(int)); w += blockDim.x) dst[w] = src[w];
  }
  if (tid == 0) {
    for (int s = 0; s < NSTAGE; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&done[s], Cfg::kGW);
      mbar_init(&empty[s], 1);
    }
    for (int h = 0; h < kGroupHelpers; ++h) issued[h] = 0;
    abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();
  const LatticeDev &L = Ls;
  if (lay_static && L.has_deps) {
    // (the host keys its graphs by has_deps: this does not happen)
    if (tid == 0) atomicExch(L.status, 1);
    return;
  }
  const int ny = L.ny, nz = L.nz, nxp = L.nxp;
  const int y_first = (L.walls & 2u) ? 1 : 0, nyf = ny - 2 * y_first;
  const int z_first = (L.walls & 4u) ? 1 : 0, nzf = nz - 2 * z_first;
  const int R = TILED ? tile_rows(PITCH, nxp) : 1;
  const int spitch = TILED ? nxp : PITCH;
  const int tpp = (nyf + R - 1) / R;
  const int ntiles = tpp * nzf;
  const unsigned limit = L.wait_limit;
  RedAcc acc;
#pragma unroll
  for (int j = 0; j < kRedWidth; ++j) acc.v[j] = 0.0;
  auto give_up = [&]() {
    if (lane == 0 && !abort_flag) {
      abort_flag = 1;
      atomicExch(L.status, 1);
    }
  };
  chain_wait();
  chain_release();

  if (warp >= kGroupConsumers) {
    // ---------------- producer h and storer h walk the block's tiles h, h + H, ...
    const int help = (warp - kGroupConsumers) >> 1;
    const bool producer = ((warp - kGroupConsumers) & 1) == 0;
    const bool withhold = L.withhold_copies != 0;
    const RowCopies rcp = row_copies(L, 2);
    // (tiles of a shorter pitch take the tiled layout: only 512 leaves a choice)
    const bool merge = TILED || PITCH == 256 || spitch == nxp;
    const CtxLane cl(lane);
    const int stride = kGroupHelpers * (int)gridDim.x, it0 = (int)blockIdx.x + help * (int)gridDim.x;
    const int step_y = stride % tpp, step_z = stride / tpp;
    int ty = it0 % tpp, tz = it0 / tpp;
    int j = help;
    Ring ring(help, NSTAGE);
    for (int it = it0; it < ntiles; it += stride, j += kGroupHelpers, ring.step(kGroupHelpers, NSTAGE)) {
      const int s = ring.s;
      unsigned char *stage = stages + s * kInStride;
      const int y0 = y_first + ty * R, z = z_first + tz, nr = min(R, nyf - ty * R);
      ty += step_y;
      tz += step_z;
      if (ty >= tpp) {
        ty -= tpp;
        ++tz;
      }
      const bool plain = plain_tile<TILED>(rcp, y0, z, nr);
      if (producer) {
        if (j >= NSTAGE && !mbar_wait_or_abort(&empty[s], ring.pass ^ 1u, limit, &abort_flag)) {
          give_up();
          break;
        }
        fill_row_ctx<RS != 0>(ctx[s], cl, y0, z, nr, ny, nz, nxp, rcp.walls, lane);
        if (lane == 0) tile_nr[s] = nr;
        __syncwarp();
        if (withhold) continue;
        const unsigned bytes = tile_bytes<LAT, __half, ODD>(nr, nxp, rcp.deps != nullptr);
        if (plain) {
          if (elect_one())
            issue_plain_tile<LAT, __half, ODD, PITCH, TILED>(rcp, smem_u32(stage), smem_u32(&full[s]), bytes, y0, z, nr, merge);
        } else {
          if (lane == 0) mbar_arrive_expect_tx(&full[s], bytes);
          __syncwarp();
          for (int b = lane; b < 64; b += 32) {
            const TileCopy c = make_tile_copy<LAT, __half, ODD, PITCH>(L, b);
            issue_tile_copy<false>(c, stage, &full[s], y0, z, nr, ny, nz, nxp, rcp.walls, spitch);
          }
        }
        __syncwarp();
        if (lane == 0) st_release(&issued[help], j / kGroupHelpers + 1);
      } else {
        if (!mbar_wait_or_abort(&done[s], ring.pass, limit, &abort_flag)) {
          give_up();
          break;
        }
        if (plain) {
          if (elect_one()) store_plain_tile<LAT, __half, ODD, PITCH, TILED>(rcp, smem_u32(stage), y0, z, nr);
        } else if (lane < LAT::Q) {
          const TileCopy c = make_tile_copy<LAT, __half, ODD, PITCH>(L, lane);
          issue_tile_copy<true>(c, stage, nullptr, y0, z, nr, ny, nz, nxp, rcp.walls, spitch);
        }
        __syncwarp();
        bulk_commit();
        bulk_wait_read<0>();  // every lane, with copies or without
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
      }
    }
    if (producer) {
      if (lane == 0 && !withhold) {
        // drain: wait (full limit) for every stage whose copies may be in
        // flight (consumers may give up after this point, too)
        for (int jj = j - kGroupHelpers; jj >= 0 && jj >= j - NSTAGE; jj -= kGroupHelpers)
          mbar_wait_bounded(&full[jj % NSTAGE], (unsigned)((jj / NSTAGE) & 1));
      }
    } else {
      bulk_wait_all();
    }
  } else {
    // ---------------- consumer groups
    const int group = warp / Cfg::kGW, gw = warp % Cfg::kGW;
    const long long n = L.n + k;
    const float dn = (float)(n - L.n_eps), dn_force = (float)(n - L.n_force);
    const bool sr = L.fp16_nearest == 0;
    // row of a position within the tile, as a multiplication (p < 256 and rows
    // of at most 128 cells where a tile has several)
    const unsigned inv = (65535u + (unsigned)nxp) / (unsigned)nxp;
    const int help = group % kGroupHelpers;  // the producer of this group's tiles
    int j = group;
    Ring ring(group, NSTAGE);
    for (int it = blockIdx.x + group * gridDim.x; it < ntiles;
         it += Cfg::kNG * gridDim.x, j += Cfg::kNG, ring.step(Cfg::kNG, NSTAGE)) {
      const int s = ring.s;
      if (!wait_issued(&issued[help], j / kGroupHelpers + 1, limit, &abort_flag) ||
          !mbar_wait_or_abort(&full[s], ring.pass, limit, &abort_flag)) {
        give_up();
        break;
      }
      unsigned char *stage = stages + s * kInStride;
      const int nr = TILED ? tile_nr[s] : 1;
#pragma unroll 1
      for (int h = 0; h < (kPair ? 1 : 2); ++h) {
        const int p = gw * 64 + (kPair ? 2 * lane : h * 32 + lane);
        const int t = TILED ? (int)((unsigned)p * inv >> 16) : 0;
        const int x = p - t * nxp;
        if (t >= nr) continue;
        const RowCtx &rc = ctx[s][t];
        // rows without a wall layer beside them (all but the first and the
        // last fluid row or plane) take the periodic code: no per-direction
        // choice of slot (D3Q27 512 x 256 x 256 with walls on y: 1.27 ms without)
        const bool at_wall = WALLS && __any_sync(__activemask(), rc.solid != 0);
        if constexpr (kPair) {
          auto go = [&](auto walls_c, auto sr_c) {
            update_row_pair<LAT, ODD, decltype(walls_c)::value, PITCH, true, decltype(sr_c)::value, TILED, RS != 0>(
                L, stage, t, rc, n, dn, dn_force, x);
          };
          if (WALLS && at_wall) {
            if (sr) go(Bool<WALLS>(), Bool<true>());
            else go(Bool<WALLS>(), Bool<false>());
          } else {
            if (sr) go(Bool<false>(), Bool<true>());
            else go(Bool<false>(), Bool<false>());
          }
        } else {
          update_row_chunk<LAT, __half, ODD, RED, WALLS, PITCH, RS, true, TILED>(L, stage, t, rc, n, dn, dn_force, x, acc);
        }
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&done[s]);
    }
  }
  __syncthreads();
  if (RED) block_reduce_store(acc, L.partials, blockIdx.x, reinterpret_cast<double(*)[kRedWidth]>(stages));
}

template <class LAT, bool W, int P, bool TL>
cudaError_t launch_group_v(const LatticeDev *L_dev, bool odd, int red, int k, const StepLaunch &ls, cudaStream_t s) {
  const int lay = (red & 4) ? 1 : 0, smem = GroupCfg<LAT, P>::kSmem;
  const dim3 grid(ls.row_grid), block(kGroupThreads);
#define LBM_GO(ODD, RED, RS) \
  return launch_chained(step_group_kernel<LAT, ODD, RED, W, P, RS, TL>, grid, block, smem, s, k > 0, L_dev, k, lay)
#define LBM_GP(RED, RS)              \
  {                                  \
    if (odd) LBM_GO(true, RED, RS);  \
    LBM_GO(false, RED, RS);          \
  }
  if (red & 1) {
    if (red & 2) LBM_GP(true, 1)
    LBM_GP(true, 0)
  }
  if (red & 2) LBM_GP(false, 1)
  LBM_GP(false, 0)
#undef LBM_GP
#undef LBM_GO
}

// ls.row as for the FP32 kernel: bit 1 walls, bit 2 pitch 512, bit 3 tiles of
// several rows
template <class LAT>
cudaError_t launch_group_t(const LatticeDev *L_dev, bool odd, int red, int k, const StepLaunch &ls, cudaStream_t s) {
  const bool w = (ls.row & 2) != 0;
  if (ls.row & 4)
    return w ? launch_group_v<LAT, true, 512, false>(L_dev, odd, red, k, ls, s)
             : launch_group_v<LAT, false, 512, false>(L_dev, odd, red, k, ls, s);
  if (ls.row & 8)
    return w ? launch_group_v<LAT, true, 256, true>(L_dev, odd, red, k, ls, s)
             : launch_group_v<LAT, false, 256, true>(L_dev, odd, red, k, ls, s);
  return w ? launch_group_v<LAT, true, 256, false>(L_dev, odd, red, k, ls, s)
           : launch_group_v<LAT, false, 256, false>(L_dev, odd, red, k, ls, s);
}

template <class LAT, bool W, int P, bool TL>
bool configure_group_v() {
  cudaError_t e = cudaSuccess;
#define LBM_CFG(ODD, RED, RS)                                                              \
  if (e == cudaSuccess)                                                                    \
  e = cudaFuncSetAttribute(step_group_kernel<LAT, ODD, RED, W, P, RS, TL>,                 \
                           cudaFuncAttributeMaxDynamicSharedMemorySize, GroupCfg<LAT, P>::kSmem)
  LBM_CFG(true, false, 0);
  LBM_CFG(true, true, 0);
  LBM_CFG(false, false, 0);
  LBM_CFG(false, true, 0);
  LBM_CFG(true, false, 1);
  LBM_CFG(true, true, 1);
  LBM_CFG(false, false, 1);
  LBM_CFG(false, true, 1);
#undef LBM_CFG
  int occ = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, step_group_kernel<LAT, true, false, W, P, 0, TL>,
                                                      kGroupThreads, GroupCfg<LAT, P>::kSmem);
  if (e != cudaSuccess) cudaGetLastError();
  return e == cudaSuccess && occ >= 1;
}

template <class LAT>
int plan_group_t(int nx, int nxp, int ny, int nz, unsigned walls, StepLaunch &ls) {
  if (nxp % 8 != 0 || nxp > 512 || nx < 8) return 0;
  if ((long long)nxp * ny * nz > 0x7fffffffLL) return 0;  // int cell indices
  if (walls & 1u) return 0;
  const bool w = (walls & 6u) != 0, p512 = nxp > 256;
  const int R = p512 ? 1 : tile_rows(256, nxp);
  const bool tl = R > 1 || (!p512 && nxp < 256);  // (one-row tiles: 28 copies instead of 38)
  bool ok;
  if (p512) ok = w ? configure_group_v<LAT, true, 512, false>() : configure_group_v<LAT, false, 512, false>();
  else if (tl) ok = w ? configure_group_v<LAT, true, 256, true>() : configure_group_v<LAT, false, 256, true>();
  else ok = w ? configure_group_v<LAT, true, 256, false>() : configure_group_v<LAT, false, 256, false>();
  const int nyf = (walls & 2u) ? ny - 2 : ny, nzf = (walls & 4u) ? nz - 2 : nz;
  if (!ok || nyf < 1 || nzf < 1) return 0;
  const long long ntiles = (long long)((nyf + R - 1) / R) * nzf;
  const int cap = sm_count();
  ls.row = 1 | (w ? 2 : 0) | (p512 ? 4 : 0) | (tl ? 8 : 0);
  ls.row_grid = ntiles < cap ? (int)ntiles : cap;
  ls.row_consumers = kGroupConsumers;
  ls.row_stages = p512 ? GroupCfg<LAT, 512>::kNS : GroupCfg<LAT, 256>::kNS;
  ls.row_smem_odd = ls.row_smem_even = 0;
  return 1;
}

}  // namespace lbm
