// Grid-side stages of one time step: the fused D2Q9 TRT collide + stream
// (a7), the step sequence, and the sorted read-outs of the bins (a2).  The
// steric and spread stages (a4-a6) are in k_steric.cu, the bead stages,
// which bin the beads, in k_bead.cu.
#include "mc_internal.cuh"

namespace mc {

// ---------------------------------------------------------------------------
// Sorted read-outs of a step's bins: the exclusive prefix sum of the bin
// counts, in blocks of kScanChunk bins (k_scan_sums adds up each block,
// k_scan_apply offsets each block by the sum of the earlier ones and scans
// it), then the records in bin order (k_sort_records).  A step does not run
// them: its tile kernels read each bin's slots directly.  They serve the
// field read-outs and saved images, and k_unsort_records puts a loaded
// image's records back into slots.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int block_sum_256(int v, int* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  int t = threadIdx.x < 8 ? red[threadIdx.x] : 0;
  if (threadIdx.x < 32) {
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) red[8] = t;
  }
  __syncthreads();
  const int r = red[8];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(256) k_scan_sums(const __grid_constant__ WorldDev w, int off) {
  __shared__ int red[9];
  const int* counts = step_counts(w, *w.t + off);
  const int base = (int)blockIdx.x * kScanChunk;
  const int end = min(base + kScanChunk, w.n_bins);
  int s = 0;
  for (int k = base + threadIdx.x; k < end; k += blockDim.x) s += counts[k];
  s = block_sum_256(s, red);
  if (threadIdx.x == 0) w.chunk_sum[blockIdx.x] = s;
}

// The offsets, and in bin_cursor each bin's first place after its slots'
// records (where k_sort_records appends the beads that found them full).
__global__ void __launch_bounds__(256) k_scan_apply(const __grid_constant__ WorldDev w, int off) {
  __shared__ int red[9];
  __shared__ int warp_tot[8];
  const int* counts = step_counts(w, *w.t + off);
  int pre = 0;
  for (int k = threadIdx.x; k < (int)blockIdx.x; k += blockDim.x) pre += w.chunk_sum[k];
  pre = block_sum_256(pre, red);
  const int n = w.n_bins;
  const int base = (int)blockIdx.x * kScanChunk + threadIdx.x * 4;
  int v[4];
  int tsum = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    v[j] = base + j < n ? counts[base + j] : 0;
    tsum += v[j];
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = tsum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  int wbase = 0;
  for (int k = 0; k < wid; ++k) wbase += warp_tot[k];
  int run = pre + wbase + incl - tsum;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int k = base + j;
    if (k < n) {
      w.bin_off[k] = run;
      w.bin_cursor[k] = run + min(v[j], w.slot_cap);
      run += v[j];
      if (k == n - 1) w.bin_off[n] = run;
    }
  }
}

// One warp per bin copies its slots; the last block appends the beads that
// found their slots full.
__global__ void __launch_bounds__(256) k_sort_records(const __grid_constant__ WorldDev w, int off) {
  const int* counts = step_counts(w, *w.t + off);
  if (blockIdx.x == gridDim.x - 1) {
    const int n = counts[w.n_bins];
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const int src = w.n_bins * w.slot_cap + k;
      const float4 p = w.bpos[src];
      const int bin = (cell_y(p) / kBin) * w.nbx + cell_x(p) / kBin;
      const int dst = atomicAdd(&w.bin_cursor[bin], 1);
      w.spos[dst] = p;
      w.srec[dst] = w.brec[src];
    }
    return;
  }
  const int bin = (int)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (bin >= w.n_bins) return;
  const int n = min(counts[bin], w.slot_cap), dst = w.bin_off[bin];
  for (int k = threadIdx.x & 31; k < n; k += 32) {
    w.spos[dst + k] = w.bpos[bin * w.slot_cap + k];
    w.srec[dst + k] = w.brec[bin * w.slot_cap + k];
  }
}

// The inverse for the last completed step (its counts start at zero).
__global__ void __launch_bounds__(256) k_unsort_records(const __grid_constant__ WorldDev w) {
  int* counts = step_counts(w, *w.t - 1);
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= w.bin_off[w.n_bins]) return;
  const float4 p = w.spos[k];
  const int bin = (cell_y(p) / kBin) * w.nbx + cell_x(p) / kBin;
  const int at = atomicAdd(&counts[bin], 1);
  const int slot = at < w.slot_cap ? bin * w.slot_cap + at : w.n_bins * w.slot_cap + atomicAdd(&counts[w.n_bins], 1);
  const float4 rec = w.srec[k];
  w.bpos[slot] = p;
  w.brec[slot] = rec;
  if (w.bead_slot) w.bead_slot[__float_as_int(rec.z)] = slot;
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
void launch_sorted_offsets(const Plan& p, cudaStream_t s, int off) {
  const WorldDev& w = p.h_world0;
  if (w.n_chunks > 1) k_scan_sums<<<w.n_chunks, 256, 0, s>>>(w, off);
  k_scan_apply<<<w.n_chunks, 256, 0, s>>>(w, off);
}

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
