// Bead-parallel stages of one time step: drive + PBD + elastic force +
// binning (a1-a3), IB interpolation + advance (a8), and
// the per-world set-up / read-out kernels.
#include <mutex>

#include "bead_dev.cuh"

namespace mc {

// a1 + a3 + a2, one warp per filament of at most 64 beads (in registers), one
// block per longer one (in dynamic shared memory): see pbd_body.
// kRoomy: twice the registers, for launches whose filaments are all resident
// at half the warps per SM (more of a filament's loads are in flight at once).
// Small launches are bound by the chain of round trips (16 filaments of 32
// beads: 7.8 us with two gathers and two claims in a row, 6.5 us so), large
// ones by how many of them are in flight and by HBM (2^22 beads: 148 us for
// some 0.6 GB, 139 us before it wrote the binned records, with 46 us of scan
// and scatter after it).
template <bool kExt, int kMode, bool kSingle, bool kLong, bool kRoomy>
__global__ void __launch_bounds__(256, kRoomy ? 2 : 4) k_pbd(const WorldDev* __restrict__ worlds,
                                             const int4* __restrict__ items, const PbdWork pw, int off,
                                             int fields) {
  pdl_trigger();
  pdl_wait();
  pbd_body<kExt, kMode, kSingle, kLong, kRoomy>(worlds, items, pw, off, fields, blockIdx.x);
}

// Spread of half of F_el + F_s at each layer point of every bead of
// two-layer worlds, in 64-bit fixed point (bitwise independent of order).
// Eight threads a bead, one stencil row of one layer point each: 10,231
// beads took 17.2 us with one thread each, 7.5 us so.
// Beads are read from the step's slots, so the positions are those at the
// start of the step even when the spread is re-run later.
__global__ void __launch_bounds__(kBeadChunk) k_layer_spread(const WorldDev* __restrict__ worlds,
                                                             const int2* __restrict__ items) {
  pdl_trigger();
  pdl_wait();
  const int2 it = items[blockIdx.x >> 3];
  const WorldDev& w = worlds[it.x];
  if (w.layers != 2) return;
  const int i = it.y + (blockIdx.x & 7) * (kBeadChunk / 8) + (threadIdx.x >> 3);
  if (i >= w.N) return;
  const int W = w.W, H = w.H;
  const int slot = w.bead_slot[i];
  if (slot < 0) return;   // no step has binned the bead
  const float4 rec = w.brec[slot];
  const float4 p = w.bpos[slot];
  const float2 n = w.nrm[i], fe = make_float2(rec.x, rec.y), fs = w.fs[i];
  const float hx = 0.5f * (fe.x + fs.x), hy = 0.5f * (fe.y + fs.y);
  const int b = threadIdx.x & 3;
  int cx, cy;
  float fx, fy;
  layer_cell(p, n, (threadIdx.x & 4) ? -w.layer_half : w.layer_half, W, H, cx, cy, fx, fy);
  float wx[4], wy[4];
  peskin4(fx, wx);
  peskin4(fy, wy);
  const float wyb = (b & 2) ? ((b & 1) ? wy[3] : wy[2]) : ((b & 1) ? wy[1] : wy[0]);
  unsigned long long* row = w.facc + 2 * (size_t)wrap_once(cy - 1 + b, H) * W;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const float g = wx[a] * wyb;
    unsigned long long* c = row + 2 * wrap_once(cx - 1 + a, W);
    // (the scale is a power of two: the products are exact)
    atomicAdd(c, (unsigned long long)__float2ll_rn(g * hx * kLayerScale));
    atomicAdd(c + 1, (unsigned long long)__float2ll_rn(g * hy * kLayerScale));
  }
}

// F = the layer spread, and the accumulator cleared for the next step.
__global__ void __launch_bounds__(kCellChunk) k_layer_finish(const WorldDev* __restrict__ worlds,
                                                             const int2* __restrict__ items) {
  pdl_trigger();
  pdl_wait();
  const int2 it = items[blockIdx.x];
  const WorldDev& w = worlds[it.x];
  if (w.layers != 2) return;
  const int c = it.y + threadIdx.x;
  if (c >= w.H * w.W) return;
  w.F[c] = layer_force(w, c);
}

// a8: U_i = sum_c delta_h(c - X_i) u(c) over the 4x4 stencil, then the
// inertia-free advance X += dt U (cell index + fraction, wrapped) and the
// unwrapped displacement D += dt U; the worlds' step counters move by inc.
template <bool kExt, bool kSingle>
__global__ void __launch_bounds__(kBeadChunk) k_interp_advance(const WorldDev* __restrict__ worlds,
                                                               const int2* __restrict__ items, int inc) {
  pdl_trigger();
  pdl_wait();
  interp_advance_body<kExt, kSingle>(worlds, items, inc, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Set-up and read-out (one world).
// ---------------------------------------------------------------------------
__constant__ int kCx[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
__constant__ int kCy[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};

// The stored state is post-collision (the LBM pulls on read).  Given
// pre-collision populations f0, store g_i(c) = f0_i(c + c_i) so that pulling
// g_i(c - c_i) returns f0_i(c).
// (A thread moves a cell's nine populations: a thread each, found by division,
// took 595 us for 4096^2; 173 us so, 1.2 GB.)
__global__ void __launch_bounds__(256) k_unstream_in(const float* __restrict__ f0, float* __restrict__ g, int H, int W) {
  pdl_trigger();
  pdl_wait();
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= W) return;
  const size_t HW = (size_t)H * W, c = (size_t)y * W + x;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    g[i * HW + c] = f0[i * HW + (size_t)wrap_once(y + kCy[i], H) * W + wrap_once(x + kCx[i], W)];
}

__global__ void __launch_bounds__(256) k_stream_out(const float* __restrict__ g, float* __restrict__ out, int H, int W) {
  pdl_trigger();
  pdl_wait();
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= W) return;
  const size_t HW = (size_t)H * W, c = (size_t)y * W + x;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    out[i * HW + c] = g[i * HW + (size_t)wrap_once(y - kCy[i], H) * W + wrap_once(x - kCx[i], W)];
}

// The bead state into device memory (any pointer may be null; nothing is
// assumed of their alignment beyond a float's).  One kernel for all four
// arrays: a small world's read-out is launches (2.6 us, where the positions'
// kernel alone took 1.9 us and the other arrays a copy each).
__global__ void __launch_bounds__(256) k_state_out(const float4* __restrict__ pos, const float2* __restrict__ disp_in,
                                                   const float* __restrict__ theta_in, int N, int E, float* x,
                                                   float* y, float* theta, float* disp) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) {
    if (x || y) {
      const float4 p = pos[i];
      if (x) x[i] = (float)cell_x(p) + p.x;
      if (y) y[i] = (float)cell_y(p) + p.y;
    }
    if (disp) {
      const float2 d = disp_in[i];
      disp[2 * (size_t)i] = d.x;
      disp[2 * (size_t)i + 1] = d.y;
    }
  }
  if (theta && i < E) theta[i] = theta_in[i];
}

// A world's set-up from its raw inputs: each position wrapped into the box
// in double precision (fmod is exact) and split into cell index + fraction,
// the creation positions, the edge angles and rest lengths, the drive records
// (theta0, A, freq, phase), the rest-length drive records (L0 = L_rest, amp,
// freq, phase), the filament offsets and the step counter.
__global__ void __launch_bounds__(256) k_world_init(const __grid_constant__ WorldDev h, const WorldRaw r) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *h.t = r.t0;
  if (i < h.N) {
    const double xd = fmod((double)r.x[i], (double)h.W), yd = fmod((double)r.y[i], (double)h.H);
    float xw = (float)(xd < 0 ? xd + h.W : xd), yw = (float)(yd < 0 ? yd + h.H : yd);
    if (xw >= (float)h.W) xw = 0.0f;
    if (yw >= (float)h.H) yw = 0.0f;
    const float cx = floorf(xw), cy = floorf(yw);
    h.pos0[i] = make_float2(xw, yw);
    h.pos[i] = make_float4(xw - cx, yw - cy, __int_as_float((int)cx), __int_as_float((int)cy));
    if (h.layers == 2) h.bead_slot[i] = -1;
  }
  if (i < h.J) const_cast<float4*>(h.drive)[i] = make_float4(r.theta0[i], r.amp[i], r.freq[i], r.phase[i]);
  if (i < h.E) {
    const float L = r.L_rest[i];
    h.theta[i] = r.theta[i];
    const_cast<float*>(h.L_rest)[i] = L;
    if (r.len_amp) const_cast<float4*>(h.ldrive)[i] = make_float4(L, r.len_amp[i], r.len_freq[i], r.len_phase[i]);
  }
  if (r.fil_off && i <= h.n_fil) const_cast<int*>(h.fil_off)[i] = r.fil_off[i];
}

__global__ void k_positions_out(const float4* __restrict__ pos, int N, float* x, float* y) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float4 p = pos[i];
  if (x) x[i] = (float)cell_x(p) + p.x;
  if (y) y[i] = (float)cell_y(p) + p.y;
}

__global__ void k_cells_out(const float4* __restrict__ pos, int N, int W, int* cell) {
  pdl_trigger();
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float4 p = pos[i];
  cell[i] = cell_y(p) * W + cell_x(p);
}

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
// Warps (filaments) per block: at most the configuration's, and few enough
// that a small launch still spreads over every SM (each warp's filament is a
// serial chain; warps sharing an SM's schedulers only delay one another).
int num_sms() {
  // first asked by kernel_setup, outside any stream capture
  static const int sms = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
  }();
  return sms;
}

struct PbdLaunch {
  PbdWork pw;
  int grid, block;
  size_t smem;
};

static PbdLaunch pbd_launch(const Plan& p) {
  const int sms = num_sms();
  const int n_short = p.n_fil_items - p.n_long;
  int wpb = p.cfg.pbd_warps;
  const int spread = (n_short + sms - 1) / sms;
  if (wpb > spread) wpb = spread;
  if (wpb < 1) wpb = 1;
  PbdLaunch l;
  l.pw.n_long = p.n_long;
  l.pw.n_items = p.n_fil_items;
  l.pw.wpb = wpb;
  l.pw.maxB = (p.max_B + 3) & ~3;
  l.grid = p.n_long + (n_short + wpb - 1) / wpb;
  l.block = wpb * 32;
  l.smem = 0;
  if (p.n_long > 0) {
    l.block = p.max_B > 128 ? 256 : 128;   // a bead or two a thread
    if (l.pw.wpb > l.block / 32) {
      l.pw.wpb = l.block / 32;
      l.grid = p.n_long + (n_short + l.pw.wpb - 1) / l.pw.wpb;
    }
    l.smem = (size_t)l.pw.maxB * kPbdFloatsPerBead * sizeof(float);
  }
  return l;
}

template <bool kExt, int kMode>
static void launch_pbd_kernel(const Plan& p, cudaStream_t s, int off, int fields) {
  if (p.n_fil_items == 0) return;
  const PbdLaunch l = pbd_launch(p);
  const bool one = p.n_worlds == 1;
  const bool roomy = !p.n_long && p.n_fil_items <= 16 * num_sms();
  auto kern = p.n_long ? (one ? k_pbd<kExt, kMode, true, true, false> : k_pbd<kExt, kMode, false, true, false>)
              : roomy  ? (one ? k_pbd<kExt, kMode, true, false, true> : k_pbd<kExt, kMode, false, false, true>)
                       : (one ? k_pbd<kExt, kMode, true, false, false> : k_pbd<kExt, kMode, false, false, false>);
  launch_pdl(kern, l.grid, l.block, l.smem, s, (const WorldDev*)p.d_worlds, (const int4*)p.d_fil_items, l.pw, off,
             fields);
}

// (worlds with a rest-length drive, observables or two layers need the
// extended kernel; it computes every other world exactly as the plain one)
void launch_pbd(const Plan& p, cudaStream_t s) {
  if (p.any_ext) launch_pbd_kernel<true, 0>(p, s, 0, 1);
  else launch_pbd_kernel<false, 0>(p, s, 0, 1);
}

// The PBD of direct-forcing worlds (from the positions the fluid carries
// the beads to; the others return at once).
void launch_pbd_mdf(const Plan& p, cudaStream_t s, int off) { launch_pbd_kernel<true, 2>(p, s, off, 1); }

// a8 of the previous step fused with this step's a1-a3 (plans without
// direct-forcing worlds), off steps after the worlds' counters.
void launch_advance_pbd(const Plan& p, cudaStream_t s, int off, int fields) {
  if (p.any_ext) launch_pbd_kernel<true, 1>(p, s, off, fields);
  else launch_pbd_kernel<false, 1>(p, s, off, fields);
}

// Shared-memory limits set once per process, outside any stream capture: the
// PBD kernel stages a filament of at most 3072 beads.
void kernel_setup() {
  static std::once_flag once;
  std::call_once(once, [] {
    steric_setup(num_sms());
    persistent_setup();
    const int most = 227 * 1024;
    for (auto f : {k_pbd<false, 0, false, true, false>, k_pbd<true, 0, false, true, false>, k_pbd<false, 1, false, true, false>,
                   k_pbd<true, 1, false, true, false>, k_pbd<true, 2, false, true, false>, k_pbd<false, 0, true, true, false>,
                   k_pbd<true, 0, true, true, false>, k_pbd<false, 1, true, true, false>, k_pbd<true, 1, true, true, false>,
                   k_pbd<true, 2, true, true, false>})
      cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  });
}

void launch_layer_spread(const Plan& p, cudaStream_t s, bool finish) {
  if (!p.any_layered) return;
  k_layer_spread<<<8 * p.n_bead_items, kBeadChunk, 0, s>>>(p.d_worlds, p.d_bead_items);
  if (finish && p.n_cell_items) k_layer_finish<<<p.n_cell_items, kCellChunk, 0, s>>>(p.d_worlds, p.d_cell_items);
}

void launch_interp_advance(const Plan& p, cudaStream_t s, int inc) {
  const bool one = p.n_worlds == 1;
  auto kern = p.any_ext ? (one ? k_interp_advance<true, true> : k_interp_advance<true, false>)
                        : (one ? k_interp_advance<false, true> : k_interp_advance<false, false>);
  launch_pdl(kern, p.n_bead_items, kBeadChunk, 0, s, p.d_worlds, p.d_bead_items, inc);
}

void launch_unstream_in(const float* f0dev, float* g_dst, int H, int W, cudaStream_t s) {
  const int nt = W < 256 ? (W + 31) & ~31 : 256;
  k_unstream_in<<<dim3((W + nt - 1) / nt, H), nt, 0, s>>>(f0dev, g_dst, H, W);
}

void launch_stream_out(const float* g_src, float* out, int H, int W, cudaStream_t s) {
  const int nt = W < 256 ? (W + 31) & ~31 : 256;
  k_stream_out<<<dim3((W + nt - 1) / nt, H), nt, 0, s>>>(g_src, out, H, W);
}

void launch_world_init(const WorldDev& w, const WorldRaw& raw, cudaStream_t s) {
  k_world_init<<<w.N / 256 + 1, 256, 0, s>>>(w, raw);   // (N >= E, J, 2 n_fil)
}

void launch_positions_out(const WorldDev& w, float* x, float* y, cudaStream_t s) {
  if (w.N == 0) return;
  k_positions_out<<<(w.N + 255) / 256, 256, 0, s>>>(w.pos, w.N, x, y);
}

void launch_state_out(const WorldDev& w, float* x, float* y, float* theta, float* disp, cudaStream_t s) {
  if (w.N == 0 || !(x || y || theta || disp)) return;
  k_state_out<<<(w.N + 255) / 256, 256, 0, s>>>(w.pos, w.disp, w.theta, w.N, w.E, x, y, theta, disp);
}

void launch_cells_out(const WorldDev& w, int* cell, cudaStream_t s) {
  if (w.N == 0) return;
  k_cells_out<<<(w.N + 255) / 256, 256, 0, s>>>(w.pos, w.N, w.W, cell);
}

}  // namespace mc
