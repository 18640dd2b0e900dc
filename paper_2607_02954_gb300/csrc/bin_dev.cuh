// Device code of the prefix sums over the bins (layout of the slots, sorted
// read-outs), shared by their kernels (k_grid.cu) and the persistent batched
// step (k_persist.cu).
#pragma once

#include "mc_internal.cuh"

namespace mc {

// ---------------------------------------------------------------------------
// Prefix sums over a world's bins, in blocks of kScanChunk bins (scan_sums
// adds up each block, scan_apply offsets each block by the sum of the earlier
// ones and scans it; worlds of one block need no sums).
//   kSrc 0  the bin counts of step (counter + off): the exclusive offsets of
//           the sorted read-outs (bin_off), and in bin_cursor each bin's first
//           place after its slots' records
//   kSrc 1  the room for the counts of the last completed step: bin_base, the
//           slots of the coming steps (left alone while no counts are in
//           place); right ahead of a step only, since no record moves
//   kSrc 2  the room for the position histogram in bin_cursor: bin_base
// The layout is by far cheaper than the sort it replaces: once in
// kLayoutSteps steps, and no record moves.  The sorted read-outs
// (k_sort_records) serve fields and saved images; k_unsort_records puts a
// loaded image's records back into slots.
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

template <int kSrc>
__device__ __forceinline__ int scan_value(const WorldDev& w, const int* counts, int k) {
  if (kSrc == 0) return counts[k];
  return slot_room(kSrc == 1 ? counts[k] : w.bin_cursor[k]);
}

struct ScanSmem {
  int red[9];
  int warp_tot[8];
};

// (block-uniform control flow: 256 threads run each whole)
template <int kSrc>
__device__ __forceinline__ void scan_sums(const WorldDev* __restrict__ worlds, const int2* __restrict__ items, int off,
                                          unsigned blk, ScanSmem& sm) {
  const int2 it = items[blk];
  const WorldDev& w = worlds[it.x];
  if (kSrc == 1 && !*w.cnt_valid) return;
  const int* counts = step_counts(w, *w.t + off);
  const int base = it.y * kScanChunk;
  const int end = min(base + kScanChunk, w.n_bins);
  int s = 0;
  for (int k = base + threadIdx.x; k < end; k += blockDim.x) s += scan_value<kSrc>(w, counts, k);
  s = block_sum_256(s, sm.red);
  if (threadIdx.x == 0) w.chunk_sum[it.y] = s;
}

template <int kSrc>
__device__ __forceinline__ void scan_apply(const WorldDev* __restrict__ worlds, const int2* __restrict__ items, int off,
                                           unsigned blk, ScanSmem& sm) {
  const int2 it = items[blk];
  const WorldDev& w = worlds[it.x];
  if (kSrc == 1 && !*w.cnt_valid) return;
  const int* counts = step_counts(w, *w.t + off);
  int pre = 0;
  for (int k = threadIdx.x; k < it.y; k += blockDim.x) pre += w.chunk_sum[k];
  pre = block_sum_256(pre, sm.red);
  const int n = w.n_bins;
  const int base = it.y * kScanChunk + threadIdx.x * 4;
  int v[4];
  int tsum = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    v[j] = base + j < n ? scan_value<kSrc>(w, counts, base + j) : 0;
    tsum += v[j];
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = tsum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) sm.warp_tot[wid] = incl;
  __syncthreads();
  int wbase = 0;
  for (int k = 0; k < wid; ++k) wbase += sm.warp_tot[k];
  int run = pre + wbase + incl - tsum;
  int* out = kSrc == 0 ? w.bin_off : w.bin_base;
  // (slot numbers stay below slot_end whatever the counts)
  auto within = [&](int r) { return kSrc == 0 || (unsigned)r <= (unsigned)w.slot_end ? r : w.slot_end; };
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int k = base + j;
    if (k < n) {
      out[k] = within(run);
      if (kSrc == 0) w.bin_cursor[k] = run + min(v[j], w.bin_base[k + 1] - w.bin_base[k]);
      run += v[j];
      if (k == n - 1) out[n] = within(run);
    }
  }
}

}  // namespace mc
