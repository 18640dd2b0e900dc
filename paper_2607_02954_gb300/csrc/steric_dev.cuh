// Device code of the steric tile stages (a4-a6) and the fused force + LBM
// tile (a5-a7), shared by the per-stage kernels (k_steric.cu) and the
// persistent batched step (k_persist.cu).  See k_steric.cu for the design.
#pragma once

#include "mc_internal.cuh"

namespace mc {

namespace {

constexpr int kThreads = 256;              // threads of a tile's block (the force kernels' narrowest, see tile_threads)
constexpr int kAx = kTile + 6;             // force accumulator edge: the tile and 3 halo cells a side
constexpr int kWin = kTile + 8;            // rho_bar window edge: the tile and 4 cells a side
__constant__ int kLbmCy[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};   // D2Q9 lattice velocities, y components

template <int R>
struct Geo {
  static constexpr int kTaps = 2 * R + 1;
  static constexpr int kL4 = (4 + 2 * R + 3) / 4;      // int4 loads per 4-column strip of the x pass
  static constexpr int kDX0 = ((kTile + 2 * R + 11 + 3) / 4) * 4;
  static constexpr int kDX1 = 4 * (kTile / 4 - 1) + 4 + 4 * kL4;
  static constexpr int kDX = kDX0 > kDX1 ? kDX0 : kDX1;   // deposit accumulator row stride (ints)
  static constexpr int kDY = kTile + 6;                    // deposit accumulator rows
  static constexpr int kLoadRows = kWin + 2 * R;           // rho_x rows staged by the force kernel
};

__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async8(void* sdst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async4(void* sdst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ int floor_div(int a, int b) { return a >= 0 ? a / b : -((b - 1 - a) / b); }

// The slots of the bins whose cells reach a cell box, as one concatenated
// list: segment e < 64 holds bin (row e / 8, column e % 8) of the box, the
// last segment the beads of the world that found their bin's slots full
// (none unless bins are crowded; each is tested against the tile like any
// other).  pre[] are the prefix sums of the segments' lengths.
constexpr int kSegs = 65;
struct Segments {
  int start[kSegs], pre[kSegs + 1];
  int covered;   // beads in the covering bins, full slots or not
  int most;      // largest bead count of one of them
};

// Builds the list for the box [x_lo, x_hi] x [y_lo, y_hi] (inclusive,
// unwrapped coordinates; at most 8 bins a side: tile + 2 R + 3 <= 51 cells)
// with one warp; lane l handles bins l and l + 32.  With kBoth the counts of
// both parities load beside the step counter that chooses between them: one
// round trip in all (force + LBM at 2^22 beads: 351 -> 337 us).  The deposit,
// whose blocks clear the other parity's counts meanwhile, loads the step's
// own after the counter (with both, 86 -> 102 us there).
template <bool kBoth>
__device__ void build_segments(const WorldDev& w, int off, int x_lo, int x_hi, int y_lo, int y_hi, Segments& sg) {
  const long long t = *w.t + off;
  const int* c0 = kBoth ? w.bin_cnt : step_counts(w, t);
  const int* c1 = w.bin_cnt + (w.n_bins + 1);
  const int lane = threadIdx.x & 31;
  const int nbx = w.nbx, nby = w.nby;
  const int* base = w.bin_base;
  int bx0 = floor_div(x_lo, kBin), bx1 = floor_div(x_hi, kBin);
  int by0 = floor_div(y_lo, kBin), by1 = floor_div(y_hi, kBin);
  if (bx1 - bx0 + 1 >= nbx) { bx0 = 0; bx1 = nbx - 1; }
  if (by1 - by0 + 1 >= nby) { by0 = 0; by1 = nby - 1; }
  const int ncol = bx1 - bx0 + 1, nrow = by1 - by0 + 1;
  const int cc = lane & 7, rr = lane >> 3;
  int lo[2] = {0, 0}, hi[2] = {0, 0}, n[2] = {0, 0}, m[2] = {0, 0};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = rr + 4 * h;
    if (cc < ncol && r < nrow) {
      const int bin = wrap_once(by0 + r, nby) * nbx + wrap_once(bx0 + cc, nbx);
      lo[h] = base[bin];
      hi[h] = base[bin + 1];
      n[h] = c0[bin];
      if (kBoth) m[h] = c1[bin];
    }
  }
  int over = c0[w.n_bins];
  const int over1 = kBoth ? c1[w.n_bins] : 0;
  if (kBoth && (t & 1)) {
    n[0] = m[0];
    n[1] = m[1];
    over = over1;
  }
  int covered = n[0] + n[1], most = max(n[0], n[1]);
  int incl0 = min(n[0], hi[0] - lo[0]), incl1 = min(n[1], hi[1] - lo[1]);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y0 = __shfl_up_sync(0xffffffffu, incl0, o), y1 = __shfl_up_sync(0xffffffffu, incl1, o);
    if (lane >= o) {
      incl0 += y0;
      incl1 += y1;
    }
  }
  incl1 += __shfl_sync(0xffffffffu, incl0, 31);
  sg.start[lane] = lo[0];
  sg.start[lane + 32] = lo[1];
  sg.pre[lane + 1] = incl0;
  sg.pre[lane + 33] = incl1;
  for (int o = 16; o > 0; o >>= 1) {
    covered += __shfl_xor_sync(0xffffffffu, covered, o);
    most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
  }
  if (lane == 31) {
    sg.pre[0] = 0;
    sg.start[kSegs - 1] = w.slot_end;
    sg.pre[kSegs] = incl1 + min(over, w.N);
    sg.covered = covered;
    sg.most = most;
  }
}

// Slot of the v-th bead of the list: the segment j with pre[j] <= v <
// pre[j + 1] by binary search over the prefix entries (non-decreasing; empty
// segments repeat a value and are never chosen).
__device__ __forceinline__ int seg_slot(int v, const Segments& sg) {
  int j = 0;
#pragma unroll
  for (int step = 32; step > 0; step >>= 1)
    if (v >= sg.pre[j + step]) j += step;
  if (j == kSegs - 2 && v >= sg.pre[kSegs - 1]) j = kSegs - 1;
  return sg.start[j] + v - sg.pre[j];
}

// Periodic image of d in (-n, n) taken in [-lo, n - lo).
__device__ __forceinline__ int image_lo(int d, int n, int lo) {
  if (d < -lo) d += n;
  else if (d >= n - lo) d -= n;
  return d;
}

// Whether r, an axis coordinate relative to the region, lies in [-lo, hi]:
// the images that reach it (and, on an axis the region covers whole, every
// cell).  For a record that the step's PBD stored the low side holds by
// construction (image_lo); one unsigned comparison checks both, so that no
// record of any bits gives an address outside the block's arrays.
__device__ __forceinline__ bool reaches(int r, int lo, int hi) { return (unsigned)(r + lo) <= (unsigned)(hi + lo); }

// The next place of the block's list for each lane that keeps its bead;
// every lane of the warp calls this together.  The list order depends on
// warp timing, which no result depends on (the accumulation is in integers).
__device__ __forceinline__ int list_place(bool keep, int* s_cnt) {
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  if (m == 0u) return 0;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(s_cnt, __popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  return base + __popc(m & ((1u << lane) - 1u));
}

template <int NT, typename T>
__device__ __forceinline__ T block_max(T v, T* red) {
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  T m = red[0];
  for (int k = 1; k < NT / 32; ++k) m = max(m, red[k]);
  __syncthreads();
  return m;
}

// The largest of the block's values.  One barrier, before the result: red is
// not written again until the block has passed another.
template <int NT>
__device__ __forceinline__ unsigned block_max_u(unsigned v, unsigned* red) {
  v = __reduce_max_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  return __reduce_max_sync(0xffffffffu, red[threadIdx.x & (NT / 32 - 1)]);
}

// The tile item of this block in a launch over the tiles of one world
// (row-major, as the plan lists them).
__device__ __forceinline__ int2 single_tile_item(const WorldDev& w, unsigned blk) {
  const unsigned ntx = (unsigned)w.ntx;
  return make_int2(0, (int)(blk % ntx) | ((int)(blk / ntx) << 16));
}

// Taps of a world with half width wR laid out for half width R >= wR.
template <int R>
__device__ __forceinline__ float padded_tap(const WorldDev& w, int wR, int m) {
  const int k = m - (R - wR);
  return (k >= 0 && k <= 2 * wR) ? w.taps[k] : 0.0f;
}

}  // namespace

// ---------------------------------------------------------------------------
// a4 + the x pass of a5.
//
// Accumulator: row ly + 3 for tile rows ly in [-3, th + 3); column
// lx + oxe for region columns lx, where the region is the tile plus wR
// columns a side (origin x0, oxe = R + 4, so every 4-column strip of the x
// pass starts on a 16-byte boundary) or, when that would cover the axis
// more than once, the whole axis (origin 0, oxe = 4, folded).
//
// The fixed-point scale 2^k comes from a bound on the cell sums: a cell's
// 4x4 stencil neighbourhood overlaps at most 2x2 bins and each bead adds at
// most 1/4, so a cell sum is below the largest bin count near the tile.
// That bound leaves at least 24 fractional bits up to about one bead per
// cell.  It is loose (a bead adds 1/16 to a cell on average), so a denser
// tile (k < 24) takes the scale that its largest sum allows (that sum plus
// the rounding its terms can hide): it deposits, measures, and deposits again
// if that scale is the finer one.  The first scale of such a tile comes from
// the beads' cells (deposit_bound, where no axis is folded): 2.25 times an
// even density's sums.  A bound known to hold may use all 32 bits of a cell
// (kWideFrom), two more than the measured rule, so this scale is as fine as the
// measured one unless a tile's sums are below a quarter of their bound, and
// hardly any tile deposits twice.
// ---------------------------------------------------------------------------

// Geometry of one deposit tile.
struct DepTile {
  int W, H, wR, x0, y0, tw, th, cx0, oxe, tile, total;
  bool full_x, full_y;
};

// Sums of a tile whose scale comes from deposit_bound fill 32 bits unsigned: b
// 2^k < 2^32 / 1.0001, and the rounding of the at most 16 b terms of a cell,
// half a unit each, adds at most 8 b < 2^15 (k >= 20 then).  Weights of rounding
// size may be negative and leave a sum some units below zero: the range above
// kWideFrom, which the other sums stay below by the 1.0001, is theirs.
// Sums that do not fit 31 bits are halved before the x pass, which reads them
// signed: that leaves one bit more than the measured rule, so the rounding of
// the halving (2^-k) and of the terms (2^-k / 2 each) stays below that rule's
// (2 2^-k a term).
constexpr unsigned kWideFrom = 0xfffe0000u;   // 2^32 - 2^17

// Deposits the tile's beads at scale 2^k into acc (zeroed) and folds the
// wrapped cells.  Ends with the block synchronised.
template <int R, int NT>
__device__ __forceinline__ void deposit_accumulate(int* acc, const WorldDev& w, const DepTile& d, int k,
                                                   const Segments& sg) {
  using G = Geo<R>;
  const int tid = threadIdx.x;
  const int W = d.W, H = d.H, wR = d.wR, x0 = d.x0, y0 = d.y0, tw = d.tw, th = d.th;
  const int cx0 = d.cx0, oxe = d.oxe, total = sg.pre[kSegs];
  const bool full_x = d.full_x, full_y = d.full_y;
  const int lo_x = full_x ? 2 : wR + 2, hi_x = full_x ? W : tw + wR;   // (the accumulator has room for both)
  const float4* __restrict__ bpos = w.bpos;
  const float scale = pow2f(k);
  // each thread deposits the beads v = tid, tid + NT, ... of the segments
  // straight from their slots, two loads in flight at a time;
  // a bead whose stencil misses the region adds nothing
  auto deposit = [&](const float4 p) {
    int rx = cell_x(p) - cx0, ry = cell_y(p) - y0;
    if (!full_x) rx = image_lo(rx, W, wR + 2);
    if (!full_y) ry = image_lo(ry, H, 2);
    if (!reaches(rx, lo_x, hi_x) || !reaches(ry, 2, th)) return;
    float wx[4], wy[4];
    peskin4(p.x, wx);
    peskin4(p.y, wy);
    int* base = acc + (ry + 2) * G::kDX + rx - 1 + oxe;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float sy = wy[b] * scale;
#pragma unroll
      for (int a = 0; a < 4; ++a) atomicAdd(base + b * G::kDX + a, __float2int_rn(wx[a] * sy));
    }
  };
  for (int v0 = tid; v0 < total; v0 += 2 * NT) {
    const int v1 = v0 + NT;
    const float4 p0 = bpos[seg_slot(v0, sg)];
    float4 p1 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (v1 < total) p1 = bpos[seg_slot(v1, sg)];
    deposit(p0);
    if (v1 < total) deposit(p1);
  }
  __syncthreads();
  if (full_x || full_y) {
    // fold the stencil cells that wrapped around an axis the region covers whole
    for (int c = tid; c < G::kDY * G::kDX; c += NT) {
      const int ly = c / G::kDX - 3, lx = c % G::kDX - oxe;
      const bool out_y = ly < 0 || ly >= th;
      const bool out_x = full_x && (lx < 0 || lx >= W);
      if ((!out_y && !out_x) || (out_y && !full_y)) continue;
      const int v = acc[c];
      if (v == 0) continue;
      const int ly2 = out_y ? wrap_mod(ly, H) : ly;
      const int lx2 = out_x ? wrap_mod(lx, W) : lx;
      atomicAdd(&acc[(ly2 + 3) * G::kDX + lx2 + oxe], v);
    }
    __syncthreads();
  }
}

// A bound of the tile's cell sums from the beads' cells alone (acc zeroed
// before, and holding the counts after): a bead of cell X adds at most
// m_a m_b / 16, m = 1, 2, 2, 1, to the cells X - 1 .. X + 2 of each axis
// (Peskin's kernel is at most 1/2 within a cell and 1/4 beyond), so a cell's
// sum is at most the weighted count of the 4 x 4 cells around it.  One atomic
// a bead instead of sixteen.  Not for folded axes.
template <int R, int NT>
__device__ __forceinline__ float deposit_bound(int* acc, const WorldDev& w, const DepTile& d, const Segments& sg,
                                               unsigned* red) {
  using G = Geo<R>;
  const int tid = threadIdx.x, total = sg.pre[kSegs];
  const float4* __restrict__ bpos = w.bpos;
  for (int v = tid; v < total; v += NT) {
    const float4 p = bpos[seg_slot(v, sg)];
    const int rx = image_lo(cell_x(p) - d.cx0, d.W, d.wR + 2), ry = image_lo(cell_y(p) - d.y0, d.H, 2);
    if (reaches(rx, d.wR + 2, d.tw + d.wR) && reaches(ry, 2, d.th)) atomicAdd(acc + (ry + 3) * G::kDX + rx + d.oxe, 1);
  }
  __syncthreads();
  int most = 0;
  for (int c = tid; c < G::kDY * G::kDX; c += NT) {
    const int i = c / G::kDX, j = c - i * G::kDX;
    int s = 0;
#pragma unroll
    for (int a = -2; a < 2; ++a) {
      if (i + a < 0 || i + a >= G::kDY) continue;
      const int* r = acc + (i + a) * G::kDX + j;
      int t = 2 * r[0];
      if (j >= 2) t += r[-2];
      if (j >= 1) t += 2 * r[-1];
      if (j + 1 < G::kDX) t += r[1];
      s += (a == -1 || a == 0) ? 2 * t : t;
    }
    most = max(most, s);
  }
  return (float)block_max_u<NT>((unsigned)most, red) * 0.0625f;
}

// The x pass of the accumulated sums at scale 2^k, rho_s when asked for,
// and the tile's bound (see k_deposit_x).
template <int R, int NT>
__device__ __forceinline__ void deposit_xpass(const int* acc, const WorldDev& w, const DepTile& d, int k,
                                              const float* tap_s, float* red, int store_fields) {
  using G = Geo<R>;
  const int tid = threadIdx.x;
  const int W = d.W, x0 = d.x0, y0 = d.y0, tw = d.tw, th = d.th, oxe = d.oxe;
  float* __restrict__ rho_x = w.rho_x;
  float* __restrict__ rho_s_out = w.rho_s;
  const float inv = pow2f(-k);
  const int col0 = x0 - d.cx0 + oxe;            // accumulator column of tile column 0
  // the tile's largest rho_s, and rho_s itself when asked for, come with the
  // x pass (the largest converted sum is the converted largest sum: the
  // conversion is monotone, and every sum is non-negative)
  float vmax = 0.0f;
  // x pass with the fixed-point scale folded into the taps (a power of two:
  // the same products as converting first)
  float tp[G::kTaps];
#pragma unroll
  for (int m = 0; m < G::kTaps; ++m) tp[m] = tap_s[m] * inv;
  if (!d.full_x) {
    const int s = tid & 7;                      // strip of 4 columns
#pragma unroll
    for (int r = 0; r < (8 * kTile + NT - 1) / NT; ++r) {
      const int ly = (tid >> 3) + r * (NT / 8);   // row
      if (ly >= th || 4 * s >= tw) continue;
      const int4* src = reinterpret_cast<const int4*>(acc + (ly + 3) * G::kDX + 4 * s + oxe - R);
      float v[4 * G::kL4];
#pragma unroll
      for (int q = 0; q < G::kL4; ++q) {
        const int4 t4 = src[q];
        v[4 * q] = (float)t4.x;
        v[4 * q + 1] = (float)t4.y;
        v[4 * q + 2] = (float)t4.z;
        v[4 * q + 3] = (float)t4.w;
      }
      float o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float sacc = 0.0f;
#pragma unroll
        for (int m = 0; m < G::kTaps; ++m) sacc = fmaf(tp[m], v[j + m], sacc);
        o[j] = sacc;
      }
      const size_t c = (size_t)(y0 + ly) * W + x0 + 4 * s;
      *reinterpret_cast<float4*>(rho_x + c) = make_float4(o[0], o[1], o[2], o[3]);
      // the strip's own cells are v[R .. R + 3]
      vmax = fmaxf(vmax, fmaxf(fmaxf(v[R], v[R + 1]), fmaxf(v[R + 2], v[R + 3])));
      if (store_fields)
        *reinterpret_cast<float4*>(rho_s_out + c) = make_float4(v[R] * inv, v[R + 1] * inv, v[R + 2] * inv, v[R + 3] * inv);
    }
  } else {
    for (int c = tid; c < th * kTile; c += NT) {
      const int ly = c >> 5, lx = c & 31;
      if (lx < tw) {
        const float v = (float)acc[(ly + 3) * G::kDX + col0 + lx];
        vmax = fmaxf(vmax, v);
        if (store_fields) rho_s_out[(size_t)(y0 + ly) * W + x0 + lx] = v * inv;
      }
    }
    for (int c = tid; c < th * tw; c += NT) {
      const int ly = c / tw, lx = c - ly * tw;
      const int* r = acc + (ly + 3) * G::kDX + oxe;
      float sacc = 0.0f;
#pragma unroll
      for (int m = 0; m < G::kTaps; ++m) sacc = fmaf(tp[m], (float)r[wrap_mod(x0 + lx - R + m, W)], sacc);
      rho_x[(size_t)(y0 + ly) * W + x0 + lx] = sacc;
    }
  }
  vmax = block_max<NT>(vmax, red);
  // Stored bound of the tile's cell sums of the kernel weights, used for
  // the fixed-point scales of the spread: the largest deposited sum plus the
  // largest rounding its terms can hide (half a unit per bead of the
  // covering bins, at most one term per cell each).  It is 0 exactly when
  // the covering bins hold no bead (written by the early exit of
  // k_deposit_x), and then no bead's stencil reaches the tile: the batched
  // force pass skips such a tile with no effect on any result.
  if (tid == 0) w.tile_rho_max[d.tile] = (vmax + 0.5f * (float)d.total) * inv;
}

// Shared memory of the deposit of one tile.
template <int R, int NT>
struct DepositSmem {
  int acc[Geo<R>::kDY * Geo<R>::kDX];
  float tap_s[Geo<R>::kTaps];
  Segments sg;
  float red[NT / 32];
  unsigned most[NT / 32];
};

// a4 + the x pass of a5 for the tile item of block `blk` (block-uniform
// control flow; the caller's block runs it whole).  It also readies the next
// step: the other parity's counts of the tile's own bins, its overflow count
// and its F_el-maximum slot go to zero (the previous step's; this step's
// stay readable).  A re-run of a completed step's deposit (off < 0) clears
// nothing: the other parity's counts may be a step's in progress.
template <int R, bool kSingle, int NT>
__device__ __forceinline__ void deposit_x_body(const WorldDev* __restrict__ worlds, const int2* __restrict__ items,
                                               int store_fields, int off, const WorldDev& w1, unsigned blk,
                                               DepositSmem<R, NT>& sm) {
  using G = Geo<R>;
  int* acc = sm.acc;
  float* tap_s = sm.tap_s;
  const Segments& sg = sm.sg;
  float* red = sm.red;
  const int2 it = kSingle ? single_tile_item(w1, blk) : items[blk];
  const WorldDev& w = kSingle ? w1 : worlds[it.x];
  DepTile d;
  d.W = w.W;
  d.H = w.H;
  d.wR = w.R;
  const int ntx = w.ntx;
  const int tx = it.y & 0xffff, ty = it.y >> 16;
  d.tile = ty * ntx + tx;
  d.x0 = tx * kTile;
  d.y0 = ty * kTile;
  d.tw = min(kTile, d.W - d.x0);
  d.th = min(kTile, d.H - d.y0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  d.full_x = d.W < d.tw + 2 * d.wR + 3;
  d.full_y = w.nty == 1;
  d.cx0 = d.full_x ? 0 : d.x0;                  // region column origin
  d.oxe = d.full_x ? 4 : R + 4;                 // accumulator column of region column 0
  if (warp == 0) build_segments<false>(w, off, d.x0 - d.wR - 2, d.x0 + d.tw + d.wR, d.y0 - 2, d.y0 + d.th, sm.sg);
  if (warp == 2 && off >= 0) {
    const long long t = *w.t + off;
    int* next = step_counts(w, t + 1);
    const int bx = d.x0 / kBin + (lane & 3), by = d.y0 / kBin + (lane >> 2);
    if (lane < 16 && bx < w.nbx && by < w.nby) next[by * w.nbx + bx] = 0;
    if (lane == 16 && d.tile == 0) {
      next[w.n_bins] = 0;
      *w.cnt_valid = 1;
      w.fel_max[(t + 1) & 1] = 0u;
    }
  }
  if (warp == 1 && lane < G::kTaps) tap_s[lane] = padded_tap<R>(w, d.wR, lane);
  for (int c = tid; c < G::kDY * G::kDX / 4; c += NT) reinterpret_cast<int4*>(acc)[c] = make_int4(0, 0, 0, 0);
  __syncthreads();
  d.total = sg.covered;
  if (d.total == 0) {
    // no bead reaches the region: rho_s, rho_x and the tile maximum are zero
    // (what the passes below give for an empty accumulator, bitwise)
    // (tw is a multiple of 8, so each 4-column strip is whole and aligned)
    const int s = tid & 7;
#pragma unroll
    for (int r = 0; r < (8 * kTile + NT - 1) / NT; ++r) {
      const int ly = (tid >> 3) + r * (NT / 8);
      if (ly >= d.th || 4 * s >= d.tw) continue;
      const size_t c = (size_t)(d.y0 + ly) * d.W + d.x0 + 4 * s;
      const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      *reinterpret_cast<float4*>(w.rho_x + c) = z;
      if (store_fields) *reinterpret_cast<float4*>(w.rho_s + c) = z;
    }
    if (tid == 0) w.tile_rho_max[d.tile] = 0.0f;
    return;
  }
  int k = fix_exponent((float)sg.most + 1.0f);
  const bool dense = k < 24;
  if (dense && !d.full_x && !d.full_y) {
    k = fix_exponent(deposit_bound<R, NT>(acc, w, d, sg, sm.most) * 1.0001f);
    if (k >= 18 && k <= 30) k += 2;   // (a term is at most 2^k / 4)
    for (int c = tid; c < G::kDY * G::kDX / 4; c += NT) reinterpret_cast<int4*>(acc)[c] = make_int4(0, 0, 0, 0);
    __syncthreads();
  }
  deposit_accumulate<R, NT>(acc, w, d, k, sg);
  if (dense) {
    // the largest accumulated sum plus the rounding of its terms
    // (half a unit per bead of the covering bins, at most one term per cell
    // each) bounds every sum; deposit again at the scale that bound gives
    unsigned m = 0u;
    auto sum = [](int v) { return (unsigned)v < kWideFrom ? (unsigned)v : 0u; };
    for (int c = tid; c < G::kDY * G::kDX / 4; c += NT) {
      const int4 v = reinterpret_cast<const int4*>(acc)[c];
      m = max(m, max(max(sum(v.x), sum(v.y)), max(sum(v.z), sum(v.w))));
    }
    m = block_max_u<NT>(m, sm.most);
    const int k2 = fix_exponent(((float)m + 0.5f * (float)d.total) * pow2f(-k) * 1.0001f);
    if (k2 > k) {
      for (int c = tid; c < G::kDY * G::kDX / 4; c += NT) reinterpret_cast<int4*>(acc)[c] = make_int4(0, 0, 0, 0);
      __syncthreads();
      k = k2;
      deposit_accumulate<R, NT>(acc, w, d, k, sg);
    } else if (m >= 0x80000000u) {
      for (int c = tid; c < G::kDY * G::kDX; c += NT) {
        const int v = acc[c];
        acc[c] = (unsigned)v < kWideFrom ? (int)(((unsigned)v + 1u) >> 1) : v / 2;
      }
      --k;
      __syncthreads();
    }
  }
  deposit_xpass<R, NT>(acc, w, d, k, tap_s, red, store_fields);
}

// ---------------------------------------------------------------------------
// The y pass of a5, and a6, for one tile; the result stays in shared memory.
//
// Window: rho_x rows [y0 - 4 - R, y0 + th + 4 + R) x columns [x0 - 4,
// x0 + tw + 4), periodic; rho_bar on window rows and columns [0, th + 8) x
// [0, tw + 8) (tile cell (lx, ly) at window (lx + 4, ly + 4)).  Spread
// accumulators: tile cell (lx, ly) at (lx + 3, ly + 3), F = acc 2^-k.
// ---------------------------------------------------------------------------
// Inputs of one tile, staged before its compute.
template <int R>
struct TileIn {
  float xb[Geo<R>::kLoadRows * kWin];   // rho_x window
  Segments sg;
  int k;                                // exponent of the spread's fixed point
  float tap_s[Geo<R>::kTaps];
};

// Beads listed per pass by a block of NT threads.
template <int NT>
constexpr int kForceCap = 5 * NT / 2;

// Working arrays of the tile being computed.
template <int NT>
struct TileWork {
  static constexpr int kCap = kForceCap<NT < kThreads ? kThreads : NT>;
  float4 sp[kCap];                      // listed beads: fractions, tile-relative cell (int bits)
  float4 sr[kCap];                      // their F_el (x, y) and bead id (int bits)
  float win[kWin * kWin];               // rho_bar window
  int accx[kAx * kAx];                  // spread accumulators
  int accy[kAx * kAx];
  int s_cnt;
};

template <int R, int NT>
struct ForceSmem {
  TileIn<R> in;
  TileWork<NT> wk;
};

struct TileBox {
  int x0, y0, tw, th;
};

// Barrier of the NT threads that run a tile's force phase: the whole block
// (NT >= kThreads), or warps 0 .. NT/32 - 1 on named barrier 1 (the
// warp-specialised kernel, whose other warps collide).
template <int NT>
__device__ __forceinline__ void force_sync() {
  if (NT >= kThreads) __syncthreads();
  else asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}

// Lists the beads c0 .. c0 + n - 1 of the tile's segments whose stencil
// reaches the tile (image taken on axes with several tiles): each thread
// reads records straight from their slots, two in flight, and the ones that
// reach the tile are packed into the working arrays.
template <int NT>
__device__ __forceinline__ void force_list(const Segments& sg, TileWork<NT>& wk, const WorldDev& w, int c0, int n,
                                           const TileBox& tb) {
  const int W = w.W, H = w.H, ntx = w.ntx, nty = w.nty;
  const float4* __restrict__ bpos = w.bpos;
  const float4* __restrict__ brec = w.brec;
  auto list = [&](bool keep, float4 p, const float4 rec) {
    int rx = cell_x(p) - tb.x0, ry = cell_y(p) - tb.y0;
    if (ntx > 1) rx = image_lo(rx, W, 2);
    if (nty > 1) ry = image_lo(ry, H, 2);
    keep = keep && reaches(rx, 2, tb.tw) && reaches(ry, 2, tb.th);
    const int at = list_place(keep, &wk.s_cnt);
    if (keep) {
      p.z = __int_as_float(rx);
      p.w = __int_as_float(ry);
      wk.sp[at] = p;
      wk.sr[at] = rec;
    }
  };
  const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  for (int v0 = 0; v0 < n; v0 += 2 * NT) {
    const int va = v0 + threadIdx.x, vb = va + NT;
    float4 pa = z, ra = z, pb = z, rb = z;
    if (va < n) {
      const int slot = seg_slot(c0 + va, sg);
      pa = bpos[slot];
      ra = brec[slot];
    }
    if (vb < n) {
      const int slot = seg_slot(c0 + vb, sg);
      pb = bpos[slot];
      rb = brec[slot];
    }
    list(va < n, pa, ra);
    if (v0 + NT < n) list(vb < n, pb, rb);   // block-uniform
  }
}

// Stage 1 of a tile: the rho_x window rows [y0 - 4 - R, y0 + th + 4 + R) x
// columns [x0 - 4, x0 + tw + 4) in 16-byte cp.async chunks (independent of
// the beads).  A 4-column chunk never straddles the periodic edge (x0 and W
// are multiples of 8); rows reach at most 4 + R <= 12 cells outside the axis.
template <int R, int NT>
__device__ __forceinline__ void tile_stage_window(TileIn<R>& in, const WorldDev& w, const TileBox& tb) {
  const int W = w.W, H = w.H, tid = threadIdx.x;
  const float* __restrict__ rho_x = w.rho_x;
  const int ww = tb.tw + 8, lh = tb.th + 8 + 2 * R;
  const int nq = ww >> 2;
  int rows_per_pass, i0;
  if (nq == kWin / 4) {   // full tile: constant divisor
    rows_per_pass = NT / (kWin / 4);
    i0 = tid / (kWin / 4);
  } else {
    rows_per_pass = NT / nq;
    i0 = tid / nq;
  }
  const int q = tid - i0 * nq;
  if (i0 < rows_per_pass) {
    const int col = wrap_once(tb.x0 - 4 + 4 * q, W);
    for (int i = i0; i < lh; i += rows_per_pass) {
      const int gy = tb.y0 - 4 - R + i;
      const int row = H >= 12 ? wrap_once(gy, H) : wrap_mod(gy, H);
      cp_async16(&in.xb[i * kWin + 4 * q], rho_x + (size_t)row * W + col);
    }
  }
}

// Stage 2 (warps 0-2, plain loads): the bead segments of the bins that reach
// the tile, the filter taps, and the largest rho_s of the 3x3 tiles around.
template <int R>
__device__ __forceinline__ void tile_stage_meta(TileIn<R>& in, const WorldDev& w, const TileBox& tb, int off) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) build_segments<true>(w, off, tb.x0 - 2, tb.x0 + tb.tw, tb.y0 - 2, tb.y0 + tb.th, in.sg);
  if (warp == 1 && lane < Geo<R>::kTaps) in.tap_s[lane] = padded_tap<R>(w, w.R, lane);
  // bound of the cell sums of weight * |F_el + F_s|:
  //   |F_s| <= k_rep/2 max|rho_bar(c+1) - rho_bar(c-1)| <= k_rep/2 max rho_bar
  //        <= k_rep/2 max rho_s over the 3x3 tiles around this one,
  // times max rho_s of this tile (the sum of the spread weights of a cell)
  if (warp == 2) {
    float v = 0.0f;   // (bounds are non-negative)
    if (lane < 9) {
      const int tx = tb.x0 / kTile, ty = tb.y0 / kTile;
      const int ty2 = wrap_once(ty + lane / 3 - 1, w.nty), tx2 = wrap_once(tx + lane % 3 - 1, w.ntx);
      v = w.tile_rho_max[ty2 * w.ntx + tx2];
    }
    const long long t = *w.t + off;
    const unsigned f0 = w.fel_max[0], f1 = w.fel_max[1];
    const float rho_max = __shfl_sync(0xffffffffu, v, 4);   // this tile's
    for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0)
      in.k = fix_exponent((__uint_as_float((t & 1) ? f1 : f0) + 0.5f * w.k_rep * v) * rho_max * 1.0001f + 1e-30f);
  }
}

// Zeroes the spread accumulators and the list count (before the barrier
// that precedes tile_compute).
template <int NT>
__device__ __forceinline__ void tile_clear(TileWork<NT>& wk) {
  for (int c = threadIdx.x; c < kAx * kAx / 4; c += NT) {
    reinterpret_cast<int4*>(wk.accx)[c] = make_int4(0, 0, 0, 0);
    reinterpret_cast<int4*>(wk.accy)[c] = make_int4(0, 0, 0, 0);
  }
  if (threadIdx.x == 0) wk.s_cnt = 0;
}

// The y pass of a5: rho_bar on the window from the staged rho_x, 8 window
// rows per thread.
template <int R, int NT>
__device__ __forceinline__ void tile_ypass(const TileIn<R>& in, TileWork<NT>& wk, const WorldDev& w, const TileBox& tb,
                                           int store_fields) {
  using G = Geo<R>;
  const int W = w.W, tw = tb.tw, th = tb.th;
  const int ww = tw + 8, wh = th + 8;
  float* __restrict__ rho_b = w.rho_b;
  float tp[G::kTaps];
#pragma unroll
  for (int m = 0; m < G::kTaps; ++m) tp[m] = in.tap_s[m];
  const int nstrip = wh >> 3;
  for (int c = threadIdx.x; c < nstrip * ww; c += NT) {
    int s;
    if (ww == kWin) s = c / kWin;   // full tile: constant divisor
    else s = c / ww;
    const int j = c - s * ww;
    const float* src = in.xb + (8 * s) * kWin + j;
    float v[8 + 2 * R];
#pragma unroll
    for (int q = 0; q < 8 + 2 * R; ++q) v[q] = src[q * kWin];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      float sacc = 0.0f;
#pragma unroll
      for (int m = 0; m < G::kTaps; ++m) sacc = fmaf(tp[m], v[r + m], sacc);
      const int i = 8 * s + r;
      wk.win[i * kWin + j] = sacc;
      if (store_fields && i >= 4 && i < th + 4 && j >= 4 && j < tw + 4)
        rho_b[(size_t)(tb.y0 + i - 4) * W + tb.x0 + j - 4] = sacc;
    }
  }
}

// a6 for the cnt listed beads: the steric force of each (kept in fs by the
// bead's own tile when asked for) and the spread of F_el + F_s into the
// accumulators at the given scale.
template <int NT>
__device__ __forceinline__ void tile_beads(TileWork<NT>& wk, const WorldDev& w, const TileBox& tb, int cnt, float scale,
                                           bool keep_fs) {
  const float k_rep = w.k_rep;
  const bool layered = w.layers == 2;
  float2* __restrict__ fs_out = w.fs;
  for (int q = threadIdx.x; q < cnt; q += NT) {
    const float4 p = wk.sp[q];
    const int rx = __float_as_int(p.z), ry = __float_as_int(p.w);
    float wx[4], wy[4];
    peskin4(p.x, wx);
    peskin4(p.y, wy);
    // stencil cell a sits at window column rx + 3 + a; the central
    // differences read one cell further on each side
    const float* base = wk.win + (ry + 2) * kWin + rx + 2;
    float gsx = 0.0f, gsy = 0.0f;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float* rowm = base + b * kWin;
      const float* row0 = rowm + kWin;
      const float* rowp = row0 + kWin;
      float sx = 0.0f, sy = 0.0f;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        sx = fmaf(wx[a], row0[a + 2] - row0[a], sx);
        sy = fmaf(wx[a], rowp[a + 1] - rowm[a + 1], sy);
      }
      gsx = fmaf(wy[b], sx, gsx);
      gsy = fmaf(wy[b], sy, gsy);
    }
    const float Fsx = -0.5f * k_rep * gsx, Fsy = -0.5f * k_rep * gsy;
    const float4 rec = wk.sr[q];
    if (keep_fs && rx >= 0 && rx < tb.tw && ry >= 0 && ry < tb.th) {
      const unsigned id = (unsigned)__float_as_int(rec.z);
      if (id < (unsigned)w.N) fs_out[id] = make_float2(Fsx, Fsy);
    }
    if (layered) continue;   // two-layer worlds spread at their layer points (k_layer_spread)
    const float Fx = (rec.x + Fsx) * scale, Fy = (rec.y + Fsy) * scale;
    float ax[4], ay[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      ax[a] = wx[a] * Fx;
      ay[a] = wx[a] * Fy;
    }
    int* bx = wk.accx + (ry + 2) * kAx + rx + 2;
    int* by = wk.accy + (ry + 2) * kAx + rx + 2;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        atomicAdd(bx + b * kAx + a, __float2int_rn(wy[b] * ax[a]));
        atomicAdd(by + b * kAx + a, __float2int_rn(wy[b] * ay[a]));
      }
    }
  }
}

// The y pass of a5 and a6 for one tile.  pull() runs once the tile's own
// loads are under way (the fused kernel starts its population reads there:
// they wait for the step counter, and nothing before needs it).  Returns k: after the caller
// synchronises the block, accx/accy hold the tile's F 2^k (before folding,
// see force_fold).
template <int R, int NT, class Pull>
__device__ __forceinline__ int force_tile(ForceSmem<R, NT>& sm, const WorldDev& w, const TileBox& tb,
                                          int store_fields, int off, bool keep_fs, Pull pull) {
  constexpr int kCap = TileWork<NT>::kCap;
  TileIn<R>& in = sm.in;
  TileWork<NT>& wk = sm.wk;
  tile_stage_window<R, NT>(in, w, tb);
  tile_stage_meta(in, w, tb, off);
  tile_clear<NT>(wk);
  pull();
  force_sync<NT>();
  const int total = in.sg.pre[kSegs];
  force_list<NT>(in.sg, wk, w, 0, min(kCap, total), tb);
  cp_async_wait_all();   // the window
  const int k = in.k;
  const float scale = pow2f(k);
  force_sync<NT>();
  // (only the beads' gradients and the rho_bar field read the y pass)
  if (total > 0 || store_fields) tile_ypass<R, NT>(in, wk, w, tb, store_fields);
  force_sync<NT>();
  tile_beads<NT>(wk, w, tb, wk.s_cnt, scale, keep_fs);
  for (int c0 = kCap; c0 < total; c0 += kCap) {
    force_sync<NT>();   // every thread is done with the previous chunk
    if (threadIdx.x == 0) wk.s_cnt = 0;
    force_sync<NT>();
    force_list<NT>(in.sg, wk, w, c0, min(kCap, total - c0), tb);
    force_sync<NT>();
    tile_beads<NT>(wk, w, tb, wk.s_cnt, scale, keep_fs);
  }
  return k;   // the caller synchronises before it reads the accumulators
}

// Folds the stencil cells that wrapped around an axis the tile covers whole
// (one tile on that axis); call after the block has synchronised.
template <int NT, class Work>
__device__ __forceinline__ void force_fold(Work& wk, const TileBox& tb, int ntx, int nty) {
  if (ntx > 1 && nty > 1) return;
  const bool fx = ntx == 1, fy = nty == 1;
  for (int c = threadIdx.x; c < kAx * kAx; c += NT) {
    const int ly = c / kAx - 3, lx = c % kAx - 3;
    const bool out_y = ly < 0 || ly >= tb.th, out_x = lx < 0 || lx >= tb.tw;
    if ((!out_y && !out_x) || (out_y && !fy) || (out_x && !fx)) continue;
    const int vx = wk.accx[c], vy = wk.accy[c];
    const int t2 = (wrap_mod(ly, tb.th) + 3) * kAx + wrap_mod(lx, tb.tw) + 3;
    if (vx) atomicAdd(&wk.accx[t2], vx);
    if (vy) atomicAdd(&wk.accy[t2], vy);
  }
  force_sync<NT>();
}

__device__ __forceinline__ TileBox tile_box(const WorldDev& w, int packed) {
  TileBox b;
  const int tx = packed & 0xffff, ty = packed >> 16;
  b.x0 = tx * kTile;
  b.y0 = ty * kTile;
  b.tw = min(kTile, w.W - b.x0);
  b.th = min(kTile, w.H - b.y0);
  return b;
}

// The tile's population rows (plane i, rows y - c_iy, 128-byte segments) to L2.
template <int NT>
__device__ __forceinline__ void prefetch_populations(const WorldDev& w, const TileBox& tb, int off) {
  const float* src = w.g[(*w.t + off) & 1];
  const int W = w.W, H = w.H;
  const size_t HW = (size_t)H * W;
  for (int c = threadIdx.x; c < 9 * kTile; c += NT) {
    const int i = c >> 5, r = c & (kTile - 1);
    if (r >= tb.th) continue;
    const int y = wrap_once(tb.y0 + r - kLbmCy[i], H);
    const float* a = src + (size_t)i * HW + (size_t)y * W + tb.x0;
    asm volatile("prefetch.global.L2 [%0];\n" ::"l"(a));
  }
}

// a7 on the tile's cells with F = acc 2^-k from shared memory.  Each warp
// collides rows warp, warp + NT / 32, ...  A warp's first row is pulled in
// begin(): by 32 warps, one row each, as soon as the tile's own loads are
// under way, so that the collision's memory round trip overlaps the force
// phase; by fewer warps, whose blocks overlap one another instead, only
// before the barrier that completes the spread (pulling earlier, or one row
// ahead in the loop, measured slower there: register pressure).
template <int NT>
struct TileLbm {
  const float* src;
  float* dst;
  int x, xm, xp, y, warp, lane;
  bool active;
  LbmPull q;

  __device__ __forceinline__ void begin(const WorldDev& w, const TileBox& tb, int off) {
    const long long t = *w.t + off;
    src = w.g[t & 1];
    dst = w.g[(t + 1) & 1];
    const int W = w.W;
    lane = threadIdx.x & 31;
    warp = threadIdx.x >> 5;
    active = lane < tb.tw && warp < tb.th;
    x = tb.x0 + lane;
    xm = x == 0 ? W - 1 : x - 1;
    xp = x == W - 1 ? 0 : x + 1;
    y = tb.y0 + warp;
    if (active) pull(w);
  }
  __device__ __forceinline__ void pull(const WorldDev& w) {
    const int W = w.W, H = w.H;
    lbm_pull(src, H * W, y * W, (y == 0 ? H - 1 : y - 1) * W, (y == H - 1 ? 0 : y + 1) * W, x, xm, xp, q);
  }
  // after the spread: synchronises the block, folds, collides
  __device__ __forceinline__ void finish(TileWork<NT>& wk, const WorldDev& w, const TileBox& tb, int k) {
    float2* __restrict__ u_out = w.u;
    const int W = w.W, HW = w.H * W;
    const LbmConst kc{w.om_p, w.om_m, w.src_p, w.src_m};
    const float inv = pow2f(-k);
    __syncthreads();
    force_fold<NT>(wk, tb, w.ntx, w.nty);
    if (!active) return;
    for (int ly = warp; ly < tb.th; ly += NT / 32) {
      if (ly != warp) pull(w);
      const int s = (ly + 3) * kAx + lane + 3;
      const float2 F = make_float2((float)wk.accx[s] * inv, (float)wk.accy[s] * inv);
      u_out[(size_t)y * W + x] = lbm_collide(q, dst, HW, y * W + x, F, kc);
      y += NT / 32;
    }
  }
};

// y pass of a5 + a6 + a7 on one tile: the force density goes from shared
// memory straight into the collision (the same arithmetic as k_force_spread
// followed by k_lbm, without F's round trip through HBM).  The tile's
// population rows are prefetched into L2 on entry, so their DRAM reads
// overlap the force phase.
template <int R, bool kSingle, int NT>
__device__ __forceinline__ void force_lbm_body(const WorldDev* __restrict__ worlds, const int2* __restrict__ items,
                                               int off, int fields, const WorldDev& w1, unsigned blk,
                                               ForceSmem<R, NT>& sm) {
  const int2 it = kSingle ? single_tile_item(w1, blk) : items[blk];
  const WorldDev& w = kSingle ? w1 : worlds[it.x];
  const TileBox tb = tile_box(w, it.y);
  const bool layered = w.layers == 2;
  const int tile = (tb.y0 / kTile) * w.ntx + tb.x0 / kTile;
  int k = 40;
  TileLbm<NT> lbm;
  constexpr bool kEarly = NT == 1024;
  if (!kSingle && !layered && w.tile_rho_max[tile] == 0.0f) {
    // no bead's stencil reaches this tile's cells (the deposit's bound is 0
    // exactly then), so it owns no bead and the spread has no term on it:
    // F = 0, as the force pass would give.  Sparse batched worlds have many
    // such tiles.
    tile_clear<NT>(sm.wk);
    lbm.begin(w, tb, off);
  } else {
    k = force_tile<R, NT>(sm, w, tb, 0, off, fields || layered, [&]() {
      if (layered) return;
      if (kEarly) lbm.begin(w, tb, off);
      else prefetch_populations<NT>(w, tb, off);
    });
    if (!kEarly && !layered) lbm.begin(w, tb, off);
  }
  // two-layer worlds: F_s only; their layer spread and collision follow in their own kernels
  if (!layered) lbm.finish(sm.wk, w, tb, k);
}

}  // namespace mc
