// a4-a6: steric deposit, Gaussian filter, steric force and immersed-boundary
// force spread, in tile kernels (one 32x32 tile of cells per block).
//
//   rho_s(c)  = sum_i delta_h(c - X_i)                        (a4, Fields)
//   rho_bar   = G_sigma * rho_s, periodic, x pass then y pass  (a5, Fields)
//   F_s,i     = -k_rep sum_c delta_h(c - X_i) grad rho_bar(c)  (a6, central differences)
//   F(c)      = sum_i delta_h(c - X_i) (F_el,i + F_s,i)       (a6, Fluid-filament Interaction)
//
// k_deposit_x    deposits rho_s on the tile plus R columns on each side in
//                shared memory, applies the x pass of the filter and writes
//                the x-filtered density rho_x of the tile (4 B per cell) and
//                a bound of the tile's rho_s (its largest deposited sum plus
//                the rounding the fixed point can hide).
// k_force_spread loads rho_x on the tile plus 4 + R rows and 4 columns,
//                applies the y pass (rho_bar on the tile plus 4 cells),
//                gathers the steric force of every bead whose stencil touches
//                the tile, spreads F_el + F_s into the tile and writes F.
// k_force_lbm    does the same and then the LBM step (a7) of the tile's
//                cells with F taken from shared memory: the step's path.
//
// The step's PBD has put every bead's record into a slot of its 8x8-cell bin,
// so the beads that can reach a tile lie in the slots of at most 8 x 8 bins.
// The force kernel stages its grid window in shared memory with cp.async,
// reads the bead records straight from their slots meanwhile and packs those
// whose stencil reaches the tile (a block-wide compaction), so its per-bead
// arithmetic runs on full warps.  The deposit, whose per-bead work is 16
// atomics, lets the beads that miss the region drop out.
//
// Both kernels are compiled for each filter half width R (1..8) so that the
// filter loops unroll with the taps in registers; a launch uses the largest R
// of its worlds, and a world with a smaller R sees its taps padded with zeros
// (which leaves every sum unchanged).  Everything that decides a result (the
// bead ranges, the fixed-point scales) uses the world's own R.
//
// Stencil cells are accumulated in a halo-extended buffer (3 cells on each
// side of the tile), so no per-cell wrap or bounds test is needed; cells
// outside the tile belong to a neighbouring tile and are dropped, except on
// an axis that one tile covers whole, where they are folded back
// periodically before use.
//
// Periodic images: with several tiles on an axis a bead is taken at the one
// image of it that can reach the tile (the reachable range is shorter than
// the axis); with one tile the tile is the whole axis.
#include <algorithm>

#include "steric_dev.cuh"

namespace mc {

// Threads of a tile's block.  A launch with fewer tiles than the SMs hold
// blocks of 256 leaves warps idle on every SM, so its tiles take wider
// blocks: 1024 threads while four times as many narrow blocks would be
// resident, 512 while twice as many would.  `regs` is the registers a thread
// of the kernel takes: 32 (deposit) or 64 (force).  A kernel that works on
// beads alone (the deposit, the spread without the collision) also wants one
// bead a thread of its tiles, else its barriers cost more than the idle
// warps (128^2, 16 tiles of 32 beads: deposit 4.7 us with 256 threads, 5.4
// with 1024).  256^2 with 4096 beads a tile: deposit 47.7 -> 24.1 us (21.6
// now that such tiles deposit once), force + LBM 53.7 -> 30.8; 512^2 with
// 1024 beads a tile: 17.1 -> 15.8 and, with 512 threads, 22.4 -> 18.9;
// 128^2: force + LBM 7.9 -> 7.1.  A tile's sums are
// integers or per-cell, so the width changes no result.
// The deposit (8.5 KB of shared memory a block) takes 128 threads from four
// tiles an SM on: sixteen tiles resident instead of eight, whose reads of
// counter, counts and records are one dependent chain, and barriers of half
// the warps.  7204 tiles of 13 beads: 25.9 -> 18.5 us, 16384 of 256 beads: 86
// -> 75, 1504: 12.4 -> 11.6, 1024: 10.0 -> 9.8; fewer leave warps idle (320
// tiles: 5.3 -> 5.5 us, 77: 5.1 -> 6.0).
int tile_threads(const Plan& p, int sms, int regs, bool beads_only) {
  const long long room = (long long)sms * (65536 / (regs * 256));   // blocks of 256 resident at once
  const long long tiles = p.n_tile_items;
  for (int nt : {1024, 512})
    if (tiles * (nt / 256) <= room && (!beads_only || p.beads >= tiles * nt)) return nt;
  if (regs == 32 && tiles >= 4 * (long long)sms) return 128;
  return 256;
}

template <int R, bool kSingle, int NT>
__global__ void __launch_bounds__(NT, 2048 / NT) k_deposit_x(const WorldDev* __restrict__ worlds,
                                                        const int2* __restrict__ items, int store_fields,
                                                        int off, const __grid_constant__ WorldDev w1) {
  pdl_trigger();
  pdl_wait();
  __shared__ __align__(16) DepositSmem<R, NT> sm;
  deposit_x_body<R, kSingle, NT>(worlds, items, store_fields, off, w1, blockIdx.x, sm);
}

// y pass of a5 + a6: writes F.  moments: direct-forcing worlds also get u* =
// (sum_i c_i f_i + F/2) / rho and rho of the tile's cells (the fluid before
// the filament's forcing), F taken from shared memory.
template <int R, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_force_spread(const WorldDev* __restrict__ worlds,
                                                           const int2* __restrict__ items, int store_fields,
                                                           int off, int moments) {
  pdl_trigger();
  pdl_wait();
  __shared__ __align__(16) ForceSmem<R, NT> sm;
  const int2 it = items[blockIdx.x];
  const WorldDev& w = worlds[it.x];
  const TileBox tb = tile_box(w, it.y);
  float2* __restrict__ F_out = w.F;
  const int W = w.W;
  const int k = force_tile<R, NT>(sm, w, tb, store_fields, off, true,
                                  [&]() { if (moments && w.ib == 1) prefetch_populations<NT>(w, tb, off); });
  __syncthreads();
  force_fold<NT>(sm.wk, tb, w.ntx, w.nty);
  const float inv = pow2f(-k);
  const int lane = threadIdx.x & 31;
  // a direct-forcing world's F holds the step's total force (steric spread
  // plus MDF passes): a re-run for the density fields leaves it
  if (store_fields && w.ib == 1) return;
  const bool mom = moments && w.ib == 1;
  const int x = tb.x0 + lane, H = w.H, HW = H * W;
  const int xm = x == 0 ? W - 1 : x - 1, xp = x == W - 1 ? 0 : x + 1;
  const float* src = mom ? w.g[(*w.t + off) & 1] : nullptr;
  float2* __restrict__ u_out = mom ? mdf_u(w, 0) : nullptr;
  for (int ly = threadIdx.x >> 5; ly < tb.th; ly += NT / 32) {
    if (lane < tb.tw) {
      const int s = (ly + 3) * kAx + lane + 3, y = tb.y0 + ly;
      const float2 F = make_float2((float)sm.wk.accx[s] * inv, (float)sm.wk.accy[s] * inv);
      const size_t c = (size_t)y * W + x;
      F_out[c] = F;
      if (mom) {
        LbmPull q;
        lbm_pull(src, HW, y * W, (y == 0 ? H - 1 : y - 1) * W, (y == H - 1 ? 0 : y + 1) * W, x, xm, xp, q);
        u_out[c] = lbm_moments(q, F, w.mrho[c]);
      }
    }
  }
}

template <int R, bool kSingle, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_force_lbm(const WorldDev* __restrict__ worlds,
                                                           const int2* __restrict__ items, int off, int fields,
                                                           const __grid_constant__ WorldDev w1) {
  pdl_trigger();
  pdl_wait();
  __shared__ __align__(16) ForceSmem<R, NT> sm;
  // tiles in reverse order: the first rows' velocities, written last, are
  // still in L2 when the next PBD (filaments in index order) interpolates
  // them, and the last rows' x-filtered densities, which the deposit wrote
  // last, are read first
  force_lbm_body<R, kSingle, NT>(worlds, items, off, fields, w1, gridDim.x - 1 - blockIdx.x, sm);
}

// y pass of a5 + a6 + a7, warp-specialised and persistent: each block walks
// the tiles blockIdx.x, blockIdx.x + gridDim.x, ...; warps 0-3 run the force
// phase of a tile (staging, y pass, steric gather, spread) while warps 4-7
// collide the previous tile, so the collision's memory traffic overlaps the
// force phase's arithmetic.  The force warps hand the tile's F over in a
// shared buffer: they fill it once the collision warps have released it
// (named barrier 4) and signal it full (named barrier 3); each tile's F and
// collision are computed exactly as in k_force_lbm (bitwise the same
// results).  Worlds without two layers only.
constexpr int kWsForce = kThreads / 2;   // threads of the force group
constexpr int kWsLbmWarps = (kThreads - kWsForce) / 32;

template <int R>
struct WsSmem {
  ForceSmem<R, kWsForce> f;
  float2 Fh[kTile * kTile];   // the hand-off buffer: F of the tile being collided
};

__device__ __forceinline__ void ws_bar_sync(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kThreads) : "memory"); }
__device__ __forceinline__ void ws_bar_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kThreads) : "memory");
}
constexpr int kWsFull = 3, kWsEmpty = 4;

template <int R, bool kSingle>
__global__ void __launch_bounds__(kThreads, 4) k_force_lbm_ws(const WorldDev* __restrict__ worlds,
                                                              const int2* __restrict__ items, int n_items, int off, int fields,
                                                              const __grid_constant__ WorldDev w1) {
  pdl_trigger();
  pdl_wait();
  extern __shared__ __align__(16) unsigned char ws_raw[];
  WsSmem<R>& sm = *reinterpret_cast<WsSmem<R>*>(ws_raw);
  const bool force_group = threadIdx.x < kWsForce;
  int done = 0;   // tiles of this block handed over so far
  for (int i = blockIdx.x; i < n_items; i += gridDim.x, ++done) {
    const int2 it = kSingle ? single_tile_item(w1, (unsigned)i) : items[i];
    const WorldDev& w = kSingle ? w1 : worlds[it.x];
    const TileBox tb = tile_box(w, it.y);
    if (force_group) {
      const int tile = (tb.y0 / kTile) * w.ntx + tb.x0 / kTile;
      int k = 40;
      if (!kSingle && w.tile_rho_max[tile] == 0.0f) {
        tile_clear<kWsForce>(sm.f.wk);   // no bead reaches the tile: F = 0 (see k_force_lbm)
      } else {
        k = force_tile<R, kWsForce>(sm.f, w, tb, 0, off, fields, [&]() { prefetch_populations<kWsForce>(w, tb, off); });
      }
      force_sync<kWsForce>();
      force_fold<kWsForce>(sm.f.wk, tb, w.ntx, w.nty);
      if (done > 0) ws_bar_sync(kWsEmpty);   // the collision warps are done with the previous F
      const float inv = pow2f(-k);
      for (int c = threadIdx.x; c < kTile * kTile; c += kWsForce) {
        const int s = ((c >> 5) + 3) * kAx + (c & 31) + 3;
        sm.Fh[c] = make_float2((float)sm.f.wk.accx[s] * inv, (float)sm.f.wk.accy[s] * inv);
      }
      force_sync<kWsForce>();   // the accumulators are read: the next tile may clear them
      ws_bar_arrive(kWsFull);
    } else {
      const int W = w.W, H = w.H, HW = H * W;
      const long long t = *w.t + off;
      const float* __restrict__ src = w.g[t & 1];
      float* __restrict__ dst = w.g[(t + 1) & 1];
      float2* __restrict__ u_out = w.u;
      const LbmConst kc{w.om_p, w.om_m, w.src_p, w.src_m};
      const int lane = threadIdx.x & 31, lw = (threadIdx.x - kWsForce) >> 5;
      const bool active = lane < tb.tw && lw < tb.th;
      const int x = tb.x0 + lane;
      const int xm = x == 0 ? W - 1 : x - 1, xp = x == W - 1 ? 0 : x + 1;
      LbmPull q;
      int y = tb.y0 + lw;
      // the first row's populations are pulled while the force warps finish
      if (active) lbm_pull(src, HW, y * W, (y == 0 ? H - 1 : y - 1) * W, (y == H - 1 ? 0 : y + 1) * W, x, xm, xp, q);
      ws_bar_sync(kWsFull);
      if (active) {
        for (int ly = lw; ly < tb.th; ly += kWsLbmWarps) {
          if (ly != lw)
            lbm_pull(src, HW, y * W, (y == 0 ? H - 1 : y - 1) * W, (y == H - 1 ? 0 : y + 1) * W, x, xm, xp, q);
          u_out[(size_t)y * W + x] = lbm_collide(q, dst, HW, y * W + x, sm.Fh[ly * kTile + lane], kc);
          y += kWsLbmWarps;
        }
      }
      ws_bar_arrive(kWsEmpty);
    }
  }
  if (force_group && done > 0) ws_bar_sync(kWsEmpty);   // the last F has been read
}

namespace {

// Blocks of the warp-specialised force + LBM kernel: as many as fit on every
// SM at once (set up outside any stream capture by steric_setup).
int g_ws_grid[kMaxR + 1] = {};
int g_sms = 1;   // (steric_setup)

template <int R>
int ws_grid() {
  return g_ws_grid[R] > 0 ? g_ws_grid[R] : 1;
}

template <int R>
void ws_setup(int sms) {
  const int bytes = (int)sizeof(WsSmem<R>);
  cudaFuncSetAttribute(k_force_lbm_ws<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(k_force_lbm_ws<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  int per = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_force_lbm_ws<R, false>, kThreads, bytes);
  g_ws_grid[R] = (per > 0 ? per : 1) * sms;
}

template <int R, int NT>
void launch_deposit(const Plan& p, cudaStream_t s, int store_fields, int off) {
  launch_pdl(p.n_worlds == 1 ? k_deposit_x<R, true, NT> : k_deposit_x<R, false, NT>, p.n_tile_items, NT, 0, s,
             p.d_worlds, p.d_tile_items, store_fields, off, p.h_world0);
}

template <int R, int NT>
void launch_spread(const Plan& p, cudaStream_t s, int store_fields, int off, int moments) {
  k_force_spread<R, NT><<<p.n_tile_items, NT, 0, s>>>(p.d_worlds, p.d_tile_items, store_fields, off, moments);
}

template <int R, int NT>
void launch_fused(const Plan& p, cudaStream_t s, int off, int fields) {
  launch_pdl(p.n_worlds == 1 ? k_force_lbm<R, true, NT> : k_force_lbm<R, false, NT>, p.n_tile_items, NT, 0, s,
             p.d_worlds, p.d_tile_items, off, fields, p.h_world0);
}

template <int R>
void launch_steric(const Plan& p, cudaStream_t s, int which, int store_fields, int off, int fields) {
  const int nt = tile_threads(p, g_sms, which == 0 ? 32 : 64, which == 0 || (which == 1 && !fields));
  if (which == 0) {
    if (nt == 1024) launch_deposit<R, 1024>(p, s, store_fields, off);
    else if (nt == 512) launch_deposit<R, 512>(p, s, store_fields, off);
    else if (nt == 128) launch_deposit<R, 128>(p, s, store_fields, off);
    else launch_deposit<R, 256>(p, s, store_fields, off);
  } else if (which == 1) {
    if (nt == 1024) launch_spread<R, 1024>(p, s, store_fields, off, fields);
    else if (nt == 512) launch_spread<R, 512>(p, s, store_fields, off, fields);
    else launch_spread<R, 256>(p, s, store_fields, off, fields);
  } else if (p.cfg.force_ws && !p.any_layered) {
    const int grid = std::min(p.n_tile_items, ws_grid<R>());
    if (p.n_worlds == 1)
      launch_pdl(k_force_lbm_ws<R, true>, grid, kThreads, sizeof(WsSmem<R>), s, p.d_worlds, p.d_tile_items,
                 p.n_tile_items, off, fields, p.h_world0);
    else
      launch_pdl(k_force_lbm_ws<R, false>, grid, kThreads, sizeof(WsSmem<R>), s, p.d_worlds, p.d_tile_items,
                 p.n_tile_items, off, fields, p.h_world0);
  } else {
    if (nt == 1024) launch_fused<R, 1024>(p, s, off, fields);
    else if (nt == 512) launch_fused<R, 512>(p, s, off, fields);
    else launch_fused<R, 256>(p, s, off, fields);
  }
}

void dispatch_steric(const Plan& p, cudaStream_t s, int which, int store_fields, int off, int fields = 1) {
  if (!p.n_tile_items) return;
  switch (p.max_R) {
    case 1: launch_steric<1>(p, s, which, store_fields, off, fields); break;
    case 2: launch_steric<2>(p, s, which, store_fields, off, fields); break;
    case 3: launch_steric<3>(p, s, which, store_fields, off, fields); break;
    case 4: launch_steric<4>(p, s, which, store_fields, off, fields); break;
    case 5: launch_steric<5>(p, s, which, store_fields, off, fields); break;
    case 6: launch_steric<6>(p, s, which, store_fields, off, fields); break;
    case 7: launch_steric<7>(p, s, which, store_fields, off, fields); break;
    default: launch_steric<kMaxR>(p, s, which, store_fields, off, fields); break;
  }
}

}  // namespace

void steric_setup(int sms) {
  g_sms = sms;
  ws_setup<1>(sms);
  ws_setup<2>(sms);
  ws_setup<3>(sms);
  ws_setup<4>(sms);
  ws_setup<5>(sms);
  ws_setup<6>(sms);
  ws_setup<7>(sms);
  ws_setup<8>(sms);
}

void launch_deposit_x(const Plan& p, cudaStream_t s, int store_fields, int off) {
  dispatch_steric(p, s, 0, store_fields, off);
}

// Two-layer worlds get F from their layer points after the tile pass.
void launch_force_spread(const Plan& p, cudaStream_t s, int store_fields, int off) {
  dispatch_steric(p, s, 1, store_fields, off, 0);
  launch_layer_spread(p, s);
}

void launch_force_moments(const Plan& p, cudaStream_t s, int off) { dispatch_steric(p, s, 1, 0, off, 1); }

void launch_force_lbm(const Plan& p, cudaStream_t s, int off, int fields) {
  dispatch_steric(p, s, 2, 0, off, fields);
  if (p.any_layered) {
    launch_layer_spread(p, s, false);
    launch_lbm(p, s, 1, off);
  }
}

}  // namespace mc
