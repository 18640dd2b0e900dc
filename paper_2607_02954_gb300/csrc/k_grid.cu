// Grid-side stages of one time step: the fused D2Q9 TRT collide + stream
// (a7), the step sequence, and the sorted read-outs of the bins (a2).  The
// steric and spread stages (a4-a6) are in k_steric.cu, the bead stages,
// which bin the beads, in k_bead.cu.
#include "bin_dev.cuh"

namespace mc {

// (see bin_dev.cuh)
template <int kSrc>
__global__ void __launch_bounds__(256) k_scan_sums(const WorldDev* __restrict__ worlds,
                                                   const int2* __restrict__ items, int off) {
  pdl_trigger();
  pdl_wait();
  __shared__ ScanSmem sm;
  scan_sums<kSrc>(worlds, items, off, blockIdx.x, sm);
}

template <int kSrc>
__global__ void __launch_bounds__(256) k_scan_apply(const WorldDev* __restrict__ worlds,
                                                    const int2* __restrict__ items, int off) {
  pdl_trigger();
  pdl_wait();
  __shared__ ScanSmem sm;
  scan_apply<kSrc>(worlds, items, off, blockIdx.x, sm);
}

// The bin of the bead at p, or -1 (a loaded image is taken as it is).
__device__ __forceinline__ int checked_bin(const WorldDev& w, const float4& p) {
  const unsigned bx = (unsigned)cell_x(p) / kBin, by = (unsigned)cell_y(p) / kBin;
  return bx < (unsigned)w.nbx && by < (unsigned)w.nby ? (int)(by * w.nbx + bx) : -1;
}

// Histogram of the beads' bins from their positions, into bin_cursor (zeroed
// before).  Once per created or loaded world; 4 us for 2^18 beads.
__global__ void __launch_bounds__(256) k_bin_histogram(const __grid_constant__ WorldDev w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= w.N) return;
  const int bin = checked_bin(w, w.pos[i]);
  if (bin >= 0) atomicAdd(&w.bin_cursor[bin], 1);
}

// The slots of a small world from its positions, in one block: the histogram
// in shared memory, then the scan of its room.  Such a world's layout is
// launches: 3.4 us at 128^2 and 512 beads, where the clearing, histogram and
// scan kernels take three launches.
constexpr int kSmallBins = 8192, kSmallBeads = 1 << 15;
__global__ void __launch_bounds__(1024) k_layout_small(const __grid_constant__ WorldDev w) {
  __shared__ int hist[kSmallBins];
  __shared__ int warp_tot[32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int k = tid; k < w.n_bins; k += 1024) hist[k] = 0;
  __syncthreads();
  for (int i = tid; i < w.N; i += 1024) {
    const int bin = checked_bin(w, w.pos[i]);
    if (bin >= 0) atomicAdd(&hist[bin], 1);
  }
  __syncthreads();
  const int per = (w.n_bins + 1023) / 1024, lo = min(tid * per, w.n_bins), hi = min(lo + per, w.n_bins);
  int sum = 0;
  for (int k = lo; k < hi; ++k) sum += slot_room(hist[k]);
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  int run = incl - sum;
  for (int k = 0; k < wid; ++k) run += warp_tot[k];
  for (int k = lo; k < hi; ++k) {
    w.bin_base[k] = run;
    run += slot_room(hist[k]);
    if (k == w.n_bins - 1) w.bin_base[k + 1] = run;
  }
}

// One warp per bin copies its slots; the last block appends the beads that
// found their slots full.
__global__ void __launch_bounds__(256) k_sort_records(const __grid_constant__ WorldDev w, int off) {
  const int* counts = step_counts(w, *w.t + off);
  if (blockIdx.x == gridDim.x - 1) {
    const int n = min(counts[w.n_bins], w.N);
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const int src = w.slot_end + k;
      const float4 p = w.bpos[src];
      const int bin = checked_bin(w, p);
      const int dst = bin < 0 ? w.N : atomicAdd(&w.bin_cursor[bin], 1);
      if (dst >= w.N) continue;   // (counts left behind by a run that timed out)
      w.spos[dst] = p;
      w.srec[dst] = w.brec[src];
    }
    return;
  }
  const int bin = (int)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (bin >= w.n_bins) return;
  const int lo = w.bin_base[bin], n = min(counts[bin], w.bin_base[bin + 1] - lo), dst = w.bin_off[bin];
  for (int k = threadIdx.x & 31; k < n && dst + k < w.N; k += 32) {
    w.spos[dst + k] = w.bpos[lo + k];
    w.srec[dst + k] = w.brec[lo + k];
  }
}

// The inverse for the last completed step (its counts start at zero).
__global__ void __launch_bounds__(256) k_unsort_records(const __grid_constant__ WorldDev w) {
  int* counts = step_counts(w, *w.t - 1);
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= w.N || k >= w.bin_off[w.n_bins]) return;
  const float4 p = w.spos[k];
  const int bin = checked_bin(w, p);
  if (bin < 0) return;
  const int at = atomicAdd(&counts[bin], 1);
  const int lo = w.bin_base[bin];
  const int slot = lo + at < w.bin_base[bin + 1] ? lo + at : w.slot_end + atomicAdd(&counts[w.n_bins], 1);
  if (k == 0) *w.cnt_valid = 1;
  const float4 rec = w.srec[k];
  w.bpos[slot] = p;
  w.brec[slot] = rec;
  const unsigned id = (unsigned)__float_as_int(rec.z);
  if (w.bead_slot && id < (unsigned)w.N) w.bead_slot[id] = slot;
}

// ---------------------------------------------------------------------------
// a7: D2Q9 lattice Boltzmann, TRT collision with Guo forcing, periodic
// streaming, fused in one pass per cell.  The state is the post-collision
// population minus the rest weight w_i (shifted storage keeps FP32 precision
// on the small deviations); a cell pulls f_i(c) = g_i(c - c_i), collides and
// stores its own post-collision populations.  With d_i = f_i - w_i:
//   rho = 1 + sum d_i,  u = (sum c_i d_i + F/2) / rho
//   feq_i - w_i = w_i [delta_rho + rho (3 c.u + 4.5 (c.u)^2 - 1.5 u.u)]
//   S_i = w_i [3 (c_i - u).F + 9 (c_i.u)(c_i.F)]
//   d*_i = d_i - (d+ - e+)/tau+ - (d- - e-)/tau- + (1 - 1/(2tau+)) S+ + (1 - 1/(2tau-)) S-
// evaluated per opposite pair (i, opp(i)) from the even and odd parts.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kCellChunk) k_lbm(const WorldDev* __restrict__ worlds,
                                                    const int2* __restrict__ items, int layered_only, int off) {
  pdl_trigger();
  pdl_wait();
  const int2 it = items[blockIdx.x];
  const WorldDev& w = worlds[it.x];
  if (layered_only && w.layers != 2) return;
  const int W = w.W, H = w.H, HW = H * W;
  const int c = it.y + threadIdx.x;
  if (c >= HW) return;
  const int y = c / W, x = c - y * W;
  const int xm = x == 0 ? W - 1 : x - 1, xp = x == W - 1 ? 0 : x + 1;
  const int ym = y == 0 ? H - 1 : y - 1, yp = y == H - 1 ? 0 : y + 1;
  const long long t = *w.t + off;
  const LbmConst k{w.om_p, w.om_m, w.src_p, w.src_m};
  // (layered_only follows the layer spread directly: its F needs no round trip through memory)
  const float2 F = layered_only ? layer_force(w, c) : w.F[c];
  w.u[c] = lbm_cell(w.g[t & 1], w.g[(t + 1) & 1], HW, y * W, ym * W, yp * W, x, xm, xp, F, k);
}

// ---------------------------------------------------------------------------
// Launchers and the step sequence.
// ---------------------------------------------------------------------------
template <int kSrc>
static void launch_scan(const Plan& p, cudaStream_t s, int off) {
  if (!p.n_scan_items) return;
  const WorldDev* ws = p.d_worlds;
  const int2* items = p.d_scan_items;
  if (!p.one_chunk) launch_pdl(k_scan_sums<kSrc>, p.n_scan_items, 256, 0, s, ws, items, off);
  launch_pdl(k_scan_apply<kSrc>, p.n_scan_items, 256, 0, s, ws, items, off);
}

void launch_slot_layout(const Plan& p, cudaStream_t s) { launch_scan<1>(p, s, -1); }

bool launch_slot_layout_small(const WorldDev& w, cudaStream_t s) {
  if (w.n_bins > kSmallBins || w.N > kSmallBeads) return false;
  k_layout_small<<<1, 1024, 0, s>>>(w);
  return true;
}

void launch_slot_layout_from_positions(const Plan& p, cudaStream_t s) {
  const WorldDev& w = p.h_world0;
  if (launch_slot_layout_small(w, s)) return;
  cudaMemsetAsync(w.bin_cursor, 0, (size_t)w.n_bins * sizeof(int), s);
  if (w.N) k_bin_histogram<<<(w.N + 255) / 256, 256, 0, s>>>(w);
  launch_scan<2>(p, s, 0);
}

void launch_sorted_offsets(const Plan& p, cudaStream_t s, int off) { launch_scan<0>(p, s, off); }

void launch_sorted_records(const Plan& p, cudaStream_t s, int off) {
  const WorldDev& w = p.h_world0;
  if (w.N) k_sort_records<<<(w.n_bins + 7) / 8 + 1, 256, 0, s>>>(w, off);
}

void launch_slots_from_sorted(const Plan& p, cudaStream_t s) {
  const WorldDev& w = p.h_world0;
  if (w.N) k_unsort_records<<<(w.N + 255) / 256, 256, 0, s>>>(w);
}

void launch_lbm(const Plan& p, cudaStream_t s, int layered_only, int off) {
  if (p.n_cell_items) k_lbm<<<p.n_cell_items, kCellChunk, 0, s>>>(p.d_worlds, p.d_cell_items, layered_only, off);
}

// n steps; in plans without direct-forcing worlds every step after the
// first runs its PBD fused with the previous step's advance (the same
// arithmetic, one kernel and one position round trip fewer), and the worlds'
// counters move by n at the end.
void enqueue_steps(const Plan& p, int n, cudaStream_t s) {
  if (p.fuse_mdf) {
    enqueue_mdf_steps(p, n, s);
    return;
  }
  if (p.any_mdf || n < 2) {
    for (int k = 0; k < n; ++k) enqueue_step(p, s);
    return;
  }
  for (int k = 0; k < n; ++k) {
    if (k == 0) launch_pbd(p, s);
    else launch_advance_pbd(p, s, k, k == n - 1);   // a8 of step k - 1 + a1-a3 of step k
    launch_deposit_x(p, s, 0, k);
    launch_force_lbm(p, s, k, k == n - 1);
  }
  launch_interp_advance(p, s, n);
}

void enqueue_step(const Plan& p, cudaStream_t s) {
  if (p.any_mdf) {
    // direct forcing: the steric spread and the MDF passes write F to device
    // memory before the LBM (the other worlds of the plan take the same
    // unfused sequence, which gives their step bitwise)
    launch_pbd(p, s);
    launch_mdf_bins(p, s);
    launch_deposit_x(p, s, 0);
    launch_force_spread(p, s, 0);
    launch_mdf(p, s);
    launch_lbm(p, s);
    launch_interp_advance(p, s);
    return;
  }
  launch_pbd(p, s);              // a1 + a3 + a2
  launch_deposit_x(p, s, 0);     // a4 + x pass of a5
  launch_force_lbm(p, s);        // y pass of a5 + a6 + a7
  launch_interp_advance(p, s);   // a8
}

}  // namespace mc
