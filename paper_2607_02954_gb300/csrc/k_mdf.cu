// Direct forcing with multi-direct-forcing (MDF) passes (Fluid-filament
// Interaction: the nodes sample the fluid velocity for their drag, the
// filament broadcasts its own velocity back onto the grid, MDF of Wang et
// al. 2008 against leakage).  For worlds with ib == 1 a step runs
//
//   k_mdf_bins      bins of X (a2) and F_el = 0, so the steric spread that
//                   follows puts only F_s on the grid (within a run fused
//                   with the previous step's advance, k_mdf_advance_bins);
//   (deposit: the penalty path's kernel)
//   k_force_spread  (k_steric.cu) the steric spread, then from F in shared
//                   memory u* = (sum_i c_i f_i + F/2) / rho and rho of every
//                   cell (the fluid before the filament's forcing);
//   k_pbd<.., 2>    X~ = X + dt I[u*](X), PBD from X~, and each bead's
//                   velocity U_s = I[u*](X) + (x_hat - X~)/dt (in ubead,
//                   and by slot in sus);
//   m passes of     k_mdf_pass, one per 32x32 tile, Jacobi in u (two buffers,
//                   see mdf_u): dF_i = 2 I[rho](X_i) (U_s,i - I[u](X_i)) for
//                   every bead whose stencil reaches the tile, the spread
//                   S[dF] in int32 fixed point (bitwise independent of
//                   order), F += S[dF] and u' = u + S[dF] / (2 rho) on the
//                   tile's cells, and F_el += dF on the bead's own tile; the
//                   last pass collides its cells with the total F at once;
//   (the advance, X^{n+1} = X + dt U_s: the penalty path's kernel).
// Plans that mix such worlds with others, or different numbers of passes,
// and the recorded steps of the reverse mode run the unfused kernels
// (k_mdf_moments, passes, k_lbm), which give the same step bitwise; there
// every kernel returns at once for the worlds of a batch that couple by the
// penalty force (and for a world's passes beyond its own m).
// Bound by the latency of each tile's phases, two waves of them at 1024
// tiles.  2^18 beads on 1024^2, us: spread with moments 29.3 (18.3 + 12.6 as
// two kernels), last pass with the collision 35 (24 + 15.9), advance with the
// bins 8.5 (7.5 + 4.2 + an idle PBD's 2.7); 16 steps of four passes 3251 ->
// 3070.  A pass alone takes 24, 22 when its records were contiguous behind a
// sort that cost 11 a step.
#include "bead_dev.cuh"
#include "steric_dev.cuh"

namespace mc {

namespace {

// a2 for a direct-forcing world's bead at p: into its bin, F_el = 0.  Every
// lane of the warp calls.
__device__ __forceinline__ void mdf_bin_bead(const WorldDev& w, int* counts, bool valid, int i, const float4 p) {
  const int bin = bead_bin_of(p, w.nbx);
  const BinClaim c = bin_claim(w, counts, valid, bin);
  if (valid) {
    w.bead_bin[i] = bin;
    w.fel[i] = make_float2(0.0f, 0.0f);
  }
  const int slot = bin_place(w, counts, valid, c);
  if (valid) bin_store(w, slot, i, p, make_float2(0.0f, 0.0f));
}

// a2 for a direct-forcing world: every bead of X into its bin (its PBD runs
// after the steric spread), and F_el = 0 (the MDF passes accumulate the bead
// forces in it).
__global__ void __launch_bounds__(kBeadChunk) k_mdf_bins(const WorldDev* __restrict__ worlds,
                                                         const int2* __restrict__ items, int off) {
  pdl_trigger();
  pdl_wait();
  const int2 it = items[blockIdx.x];
  const WorldDev& w = worlds[it.x];
  if (w.ib != 1) return;
  const int i = it.y + threadIdx.x;
  const bool valid = i < w.N;
  mdf_bin_bead(w, step_counts(w, *w.t + off), valid, i, valid ? w.pos[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f));
}

// a8 of the previous step (X += dt U_s) and the bins of this one.
__global__ void __launch_bounds__(kBeadChunk) k_mdf_advance_bins(const WorldDev* __restrict__ worlds,
                                                                 const int2* __restrict__ items, int off) {
  pdl_trigger();
  pdl_wait();
  const int2 it = items[blockIdx.x];
  const WorldDev& w = worlds[it.x];
  const int i = it.y + threadIdx.x;
  const bool valid = i < w.N;
  float4 p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float2 d = make_float2(0.0f, 0.0f), U = d;
  long long q = 0;
  if (valid) {
    p = w.pos[i];
    d = w.disp[i];
    U = w.ubead[i];
    bead_energy(w, i, p, q);
  }
  if (w.observe && w.energy) obs_add_warp(&w.obs[2], q);
  if (valid) p = advance_tail<false>(w, w.u_max, i, p, d, U.x, U.y);
  mdf_bin_bead(w, step_counts(w, *w.t + off), valid, i, p);
}

// u* and rho of every cell from the pulled populations and the steric F.
__global__ void __launch_bounds__(kCellChunk) k_mdf_moments(const WorldDev* __restrict__ worlds,
                                                            const int2* __restrict__ items) {
  pdl_trigger();
  pdl_wait();
  const int2 it = items[blockIdx.x];
  const WorldDev& w = worlds[it.x];
  if (w.ib != 1) return;
  const int W = w.W, H = w.H, HW = H * W;
  const int c = it.y + threadIdx.x;
  if (c >= HW) return;
  const int y = c / W, x = c - y * W;
  const int xm = x == 0 ? W - 1 : x - 1, xp = x == W - 1 ? 0 : x + 1;
  const int ym = y == 0 ? H - 1 : y - 1, yp = y == H - 1 ? 0 : y + 1;
  LbmPull q;
  lbm_pull(w.g[*w.t & 1], HW, y * W, ym * W, yp * W, x, xm, xp, q);
  const float2 F = w.F[c];
  mdf_u(w, 0)[c] = lbm_moments(q, F, w.mrho[c]);
}

// One MDF pass of the direct-forcing worlds on one tile, Jacobi in u.  Every
// bead whose stencil reaches the tile gets
//   dF_i = 2 I[rho](X_i) (U_s,i - I[u](X_i))
// from the pass's input velocity and rho, both staged with a 3-cell halo;
// then the tile's cells get F += S[dF] and u' = u + S[dF] / (2 rho) in the
// other velocity buffer, and with `fields` the tile that holds a bead adds its
// dF to F_el.  A bead near a tile edge is evaluated by each tile its stencil
// reaches, from the same inputs in the same order, so every tile uses the
// same dF bitwise.  The spread is in int32 fixed point with the scale from
// the largest |dF| component among the tile's beads times the tile's largest
// rho_s (the sum of the spread weights of a cell): bitwise independent of
// order.  The dF of a tile's beads are kept in shared memory when they fit
// one pass over the list, and are evaluated again in a second sweep
// otherwise.
// With `fuse` a world's last pass hands F straight to the collision of its
// cells (its u' would not be read; F is kept with `fields`).
constexpr int kMwy = kTile + 6;   // window rows: the tile and 3 cells a side
constexpr int kMwx = kTile + 8;   // window columns: the tile and 4 cells a side (16-byte chunks)

template <int NT>
struct MdfSmem {
  static constexpr int kCap = kForceCap<NT>;
  float4 sp[kCap];          // listed beads: fractions, tile-relative cell (int bits)
  float2 su[kCap];          // their U_s
  float2 df[kCap];          // their dF (one-list tiles)
  int si[kCap];             // their bead indices
  float2 uw[kMwy * kMwx];   // input velocity window
  float rw[kMwy * kMwx];    // density window
  int accx[kAx * kAx];      // spread accumulators
  int accy[kAx * kAx];
  int s_cnt;
  Segments sg;
  float red[NT / 32];
};

// dF of listed bead v: its stencil cells sit at window rows ry + 2 .. ry + 5
// and columns rx + 3 .. rx + 6.
template <int NT>
__device__ __forceinline__ float2 mdf_bead_force(const MdfSmem<NT>& sm, int v) {
  const float4 p = sm.sp[v];
  const int rx = __float_as_int(p.z), ry = __float_as_int(p.w);
  float wx[4], wy[4];
  peskin4(p.x, wx);
  peskin4(p.y, wy);
  float Ux = 0.0f, Uy = 0.0f, r = 0.0f;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int row = (ry + 2 + b) * kMwx + rx + 3;
    float ax = 0.0f, ay = 0.0f, ar = 0.0f;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float2 v2 = sm.uw[row + a];
      ax = fmaf(wx[a], v2.x, ax);
      ay = fmaf(wx[a], v2.y, ay);
      ar = fmaf(wx[a], sm.rw[row + a], ar);
    }
    Ux = fmaf(wy[b], ax, Ux);
    Uy = fmaf(wy[b], ay, Uy);
    r = fmaf(wy[b], ar, r);
  }
  const float2 Us = sm.su[v];
  return make_float2(2.0f * r * (Us.x - Ux), 2.0f * r * (Us.y - Uy));
}

// Lists the beads c0 .. c0 + n - 1 of the tile's segments whose stencil
// reaches the tile, straight from their slots, two records in flight a
// thread (as force_list).
template <int NT>
__device__ __forceinline__ void mdf_list(MdfSmem<NT>& sm, const WorldDev& w, const TileBox& tb, int c0, int n) {
  struct Rec {
    float4 p;
    float2 us;
    int id;
  };
  auto load = [&](int v) {
    Rec r;
    r.p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    r.us = make_float2(0.0f, 0.0f);
    r.id = 0;
    if (v < n) {
      const int slot = seg_slot(c0 + v, sm.sg);
      r.p = w.bpos[slot];
      r.us = w.sus[slot];
      r.id = __float_as_int(w.brec[slot].z);
    }
    return r;
  };
  auto list = [&](bool keep, Rec r) {
    int rx = cell_x(r.p) - tb.x0, ry = cell_y(r.p) - tb.y0;
    if (w.ntx > 1) rx = image_lo(rx, w.W, 2);
    if (w.nty > 1) ry = image_lo(ry, w.H, 2);
    keep = keep && reaches(rx, 2, tb.tw) && reaches(ry, 2, tb.th);
    const int at = list_place(keep, &sm.s_cnt);
    if (keep) {
      r.p.z = __int_as_float(rx);
      r.p.w = __int_as_float(ry);
      sm.sp[at] = r.p;
      sm.su[at] = r.us;
      sm.si[at] = r.id;
    }
  };
  for (int v0 = 0; v0 < n; v0 += 2 * NT) {
    const int va = v0 + threadIdx.x;
    const Rec ra = load(va), rb = load(va + NT);
    list(va < n, ra);
    if (v0 + NT < n) list(va + NT < n, rb);   // block-uniform
  }
}

template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_mdf_pass(const WorldDev* __restrict__ worlds,
                                                            const int2* __restrict__ items, int pass, int off,
                                                            int fields, int fuse) {
  pdl_trigger();
  pdl_wait();
  __shared__ __align__(16) MdfSmem<NT> sm;
  constexpr int kCap = MdfSmem<NT>::kCap;
  const int2 it = items[blockIdx.x];
  const WorldDev& w = worlds[it.x];
  if (w.ib != 1 || pass >= w.mdf_iters) return;
  const bool collide = fuse && pass == w.mdf_iters - 1;
  const TileBox tb = tile_box(w, it.y);
  const int W = w.W, H = w.H, ntx = w.ntx, nty = w.nty;
  const int tile = (tb.y0 / kTile) * ntx + tb.x0 / kTile;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float2* __restrict__ u_in = mdf_u(w, pass);
  if (warp == 0) build_segments<true>(w, off, tb.x0 - 2, tb.x0 + tb.tw, tb.y0 - 2, tb.y0 + tb.th, sm.sg);
  // the velocity and density windows, rows y0 - 3 .. y0 + th + 2 and
  // columns x0 - 4 .. x0 + tw + 3, periodic (W, H >= 8: one wrap at most),
  // in 16-byte chunks (2 velocities or 4 densities; x0 and W are multiples
  // of 8, so a chunk never straddles the periodic edge)
  const bool full = tb.tw == kTile;   // full tile: constant divisors
  const int nu = full ? kMwx / 2 : (tb.tw + 8) >> 1, nr = full ? kMwx / 4 : (tb.tw + 8) >> 2, wh = tb.th + 6;
  for (int c = tid; c < wh * nu; c += NT) {
    const int i = full ? c / (kMwx / 2) : c / nu, j = 2 * (c - i * nu);
    const size_t g = (size_t)wrap_once(tb.y0 - 3 + i, H) * W + wrap_once(tb.x0 - 4 + j, W);
    cp_async16(&sm.uw[i * kMwx + j], &u_in[g]);
  }
  for (int c = tid; c < wh * nr; c += NT) {
    const int i = full ? c / (kMwx / 4) : c / nr, j = 4 * (c - i * nr);
    const size_t g = (size_t)wrap_once(tb.y0 - 3 + i, H) * W + wrap_once(tb.x0 - 4 + j, W);
    cp_async16(&sm.rw[i * kMwx + j], &w.mrho[g]);
  }
  for (int c = tid; c < kAx * kAx / 4; c += NT) {
    reinterpret_cast<int4*>(sm.accx)[c] = make_int4(0, 0, 0, 0);
    reinterpret_cast<int4*>(sm.accy)[c] = make_int4(0, 0, 0, 0);
  }
  if (tid == 0) sm.s_cnt = 0;
  if (collide) prefetch_populations<NT>(w, tb, off);
  __syncthreads();   // segments visible
  const int total = sm.sg.pre[kSegs];
  const bool one_list = total <= kCap;
  // sweep 1: dF of every listed bead and their largest component
  float m = 0.0f;
  for (int c0 = 0; c0 < total; c0 += kCap) {
    if (c0 > 0) {
      __syncthreads();   // the previous list is no longer read
      if (tid == 0) sm.s_cnt = 0;
      __syncthreads();
    }
    mdf_list<NT>(sm, w, tb, c0, min(kCap, total - c0));
    cp_async_wait_all();   // the windows, the first time
    __syncthreads();
    const int cnt = sm.s_cnt;
    for (int q = tid; q < cnt; q += NT) {
      const float2 dF = mdf_bead_force<NT>(sm, q);
      if (one_list) sm.df[q] = dF;
      m = fmaxf(m, fmaxf(fabsf(dF.x), fabsf(dF.y)));
    }
  }
  if (total == 0) cp_async_wait_all();
  // the warp's rows warp, warp + NT / 32, ...: every F load in flight during the spread
  float2* __restrict__ Fg = w.F;
  constexpr int kRows = kTile / (NT / 32);
  float2 Fv[kRows];
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    const int ly = warp + r * (NT / 32);
    if (ly < tb.th && lane < tb.tw) Fv[r] = Fg[(size_t)(tb.y0 + ly) * W + tb.x0 + lane];
  }
  m = block_max<NT>(m, sm.red);   // also orders the df writes before sweep 2
  const int k = fix_exponent(m * w.tile_rho_max[tile] * 1.0001f + 1e-30f);
  const float scale = pow2f(k);
  // sweep 2: the spread, and F_el += dF on the bead's own tile
  float2* __restrict__ fel = w.fel;
  for (int c0 = 0; c0 < total; c0 += kCap) {
    if (!one_list) {
      __syncthreads();
      if (tid == 0) sm.s_cnt = 0;
      __syncthreads();
      mdf_list<NT>(sm, w, tb, c0, min(kCap, total - c0));
      __syncthreads();
    }
    const int cnt = sm.s_cnt;
    for (int q = tid; q < cnt; q += NT) {
      const float2 dF = one_list ? sm.df[q] : mdf_bead_force<NT>(sm, q);
      const float4 p = sm.sp[q];
      const int rx = __float_as_int(p.z), ry = __float_as_int(p.w);
      if (fields && rx >= 0 && rx < tb.tw && ry >= 0 && ry < tb.th) {
        // the bead's own tile is its one writer in this pass: the adds
        // need no return value and leave the same bits in any order
        const int i = sm.si[q];
        if ((unsigned)i < (unsigned)w.N) {
          atomicAdd(&fel[i].x, dF.x);
          atomicAdd(&fel[i].y, dF.y);
        }
      }
      float wx[4], wy[4];
      peskin4(p.x, wx);
      peskin4(p.y, wy);
      const float Fx = dF.x * scale, Fy = dF.y * scale;
      int* bx = sm.accx + (ry + 2) * kAx + rx + 2;
      int* by = sm.accy + (ry + 2) * kAx + rx + 2;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const float g = wx[a] * wy[b];
          atomicAdd(bx + b * kAx + a, __float2int_rn(g * Fx));
          atomicAdd(by + b * kAx + a, __float2int_rn(g * Fy));
        }
      }
    }
  }
  __syncthreads();
  force_fold<NT>(sm, tb, ntx, nty);
  const float inv = pow2f(-k);
  float2* __restrict__ u_out = mdf_u(w, pass + 1);
  const int x = tb.x0 + lane, HW = H * W;
  const int xm = x == 0 ? W - 1 : x - 1, xp = x == W - 1 ? 0 : x + 1;
  const long long t = collide ? *w.t + off : 0;
  const float* src = w.g[t & 1];
  float* dst = w.g[(t + 1) & 1];
  const LbmConst kc{w.om_p, w.om_m, w.src_p, w.src_m};
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    const int ly = warp + r * (NT / 32);
    if (ly < tb.th && lane < tb.tw) {
      const int sidx = (ly + 3) * kAx + lane + 3;
      const int widx = (ly + 3) * kMwx + lane + 4;
      const int y = tb.y0 + ly;
      const size_t c = (size_t)y * W + x;
      const float Gx = (float)sm.accx[sidx] * inv, Gy = (float)sm.accy[sidx] * inv;
      const float2 F = make_float2(Fv[r].x + Gx, Fv[r].y + Gy);
      if (!collide || fields) Fg[c] = F;
      if (collide) {
        u_out[c] = lbm_cell(src, dst, HW, y * W, (y == 0 ? H - 1 : y - 1) * W, (y == H - 1 ? 0 : y + 1) * W, x, xm, xp,
                            F, kc);
      } else {
        const float ih = __frcp_rn(2.0f * sm.rw[widx]);   // 1 / (2 rho), correctly rounded
        const float2 u = sm.uw[widx];
        u_out[c] = make_float2(fmaf(Gx, ih, u.x), fmaf(Gy, ih, u.y));
      }
    }
  }
}

}  // namespace

void launch_pbd_mdf(const Plan& p, cudaStream_t s, int off);   // k_bead.cu

void launch_mdf_bins(const Plan& p, cudaStream_t s, int off) {
  if (!p.any_mdf) return;
  k_mdf_bins<<<p.n_bead_items, kBeadChunk, 0, s>>>(p.d_worlds, p.d_bead_items, off);
}

// (the block's width as for the fused force + LBM kernel, see tile_threads)
void launch_mdf_pass(const Plan& p, cudaStream_t s, int pass, int off, int fields, int fuse) {
  if (!p.n_tile_items) return;
  const int nt = tile_threads(p, num_sms(), 64, false);
  auto kern = nt == 1024 ? k_mdf_pass<1024> : nt == 512 ? k_mdf_pass<512> : k_mdf_pass<256>;
  launch_pdl(kern, p.n_tile_items, nt, 0, s, (const WorldDev*)p.d_worlds, (const int2*)p.d_tile_items, pass, off,
             fields, fuse);
}

void launch_mdf(const Plan& p, cudaStream_t s) {
  if (!p.any_mdf) return;
  if (p.n_cell_items) k_mdf_moments<<<p.n_cell_items, kCellChunk, 0, s>>>(p.d_worlds, p.d_cell_items);
  launch_pbd_mdf(p, s, 0);
  for (int k = 0; k < p.max_mdf; ++k) launch_mdf_pass(p, s, k, 0, 1, 0);
}

void enqueue_mdf_steps(const Plan& p, int n, cudaStream_t s) {
  for (int k = 0; k < n; ++k) {
    if (k == 0) launch_mdf_bins(p, s, 0);
    else launch_pdl(k_mdf_advance_bins, p.n_bead_items, kBeadChunk, 0, s, (const WorldDev*)p.d_worlds,
                    (const int2*)p.d_bead_items, k);
    launch_deposit_x(p, s, 0, k);
    launch_force_moments(p, s, k);
    launch_pbd_mdf(p, s, k);
    for (int j = 0; j < p.max_mdf; ++j) launch_mdf_pass(p, s, j, k, k == n - 1, 1);
  }
  launch_interp_advance(p, s, n);
}

// launch_mdf for the one world h of plan p, keeping u_0 (the drag's
// velocity) and each pass's input velocity (u_0 .. u_{m-1}, m =
// h.mdf_iters) in mu[k H W ..] for the reverse mode.
cudaError_t launch_mdf_recorded(const Plan& p, const WorldDev& h, float2* mu, cudaStream_t s) {
  const size_t bytes = (size_t)h.H * h.W * sizeof(float2);
  if (p.n_cell_items) k_mdf_moments<<<p.n_cell_items, kCellChunk, 0, s>>>(p.d_worlds, p.d_cell_items);
  cudaError_t e = cudaSuccess;
  e = cudaMemcpyAsync(mu, mdf_u(h, 0), bytes, cudaMemcpyDeviceToDevice, s);
  launch_pbd_mdf(p, s, 0);
  for (int k = 0; k < h.mdf_iters && e == cudaSuccess; ++k) {
    launch_mdf_pass(p, s, k, 0, 1, 0);
    if (k + 1 < h.mdf_iters)
      e = cudaMemcpyAsync(reinterpret_cast<char*>(mu) + (k + 1) * bytes, mdf_u(h, k + 1), bytes,
                          cudaMemcpyDeviceToDevice, s);
  }
  return e;
}

}  // namespace mc
