// Device code of the bead-parallel stages (a1-a3 PBD with a2's binning, a8
// interpolation + advance), shared by the per-stage kernels (k_bead.cu) and
// the persistent batched step (k_persist.cu).
#pragma once

#include "mc_internal.cuh"

namespace mc {

constexpr int kPbdFloatsPerBead = 18;

__device__ __forceinline__ void cpa16(void* sdst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cpa4(void* sdst, const void* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cpa_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }


// X + dt U in cell + fraction form, wrapped, for X = p.
__device__ __forceinline__ float4 advance_pos(const WorldDev& w, float4 p, float Ux, float Uy) {
  const int W = w.W, H = w.H;
  int cx = cell_x(p), cy = cell_y(p);
  float fx = p.x + w.dt * Ux, fy = p.y + w.dt * Uy;
  const float kx = floorf(fx), ky = floorf(fy);
  fx -= kx;
  fy -= ky;
  cx += (int)kx;
  cy += (int)ky;
  if (fx >= 1.0f) { fx = 0.0f; cx += 1; }   // a tiny negative fraction rounded up to 1
  if (fy >= 1.0f) { fy = 0.0f; cy += 1; }
  cx = wrap_once(cx, W);
  cy = wrap_once(cy, H);
  return make_float4(fx, fy, __int_as_float(cx), __int_as_float(cy));
}

// a8 for one bead at p = X^n with velocity U: the velocity record (kRecord;
// the advance fused into the next step's PBD skips it, since a run of steps
// ends with a standalone advance that writes the last step's), the watchdog
// (|U| > u_max or non-finite: flag the world, keep the bead),
// X^{n+1} = wrap(X^n + dt U) in cell + fraction form, D += dt U.
// Returns X^{n+1} (X^n when the watchdog fired).
// d: the bead's displacement so far.
template <bool kRecord = true>
__device__ __forceinline__ float4 advance_tail(const WorldDev& w, float u_max, int i, float4 p, float2 d, float Ux,
                                               float Uy) {
  if (kRecord) w.ubead[i] = make_float2(Ux, Uy);
  const float m2 = Ux * Ux + Uy * Uy;
  if (!(m2 <= u_max * u_max)) {   // also catches NaN
    atomicOr(w.flags, kFlagUnstable);
    return p;
  }
  const float4 q = advance_pos(w, p, Ux, Uy);
  w.pos[i] = q;
  d.x += w.dt * Ux;
  d.y += w.dt * Uy;
  w.disp[i] = d;
  return q;
}

// U_i = sum_c delta_h(c - X_i) u(c) over the 4x4 stencil of p, for the
// velocity field u of a W x H grid.
__device__ __forceinline__ float2 interp_field(const float2* __restrict__ u, int W, int H, const float4 p) {
  const int cx = cell_x(p), cy = cell_y(p);
  float wx[4], wy[4];
  peskin4(p.x, wx);
  peskin4(p.y, wy);
  int ix[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) ix[a] = wrap_once(cx - 1 + a, W);
  float Ux = 0.0f, Uy = 0.0f;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const float2* row = u + (size_t)wrap_once(cy - 1 + b, H) * W;
    float rx = 0.0f, ry = 0.0f;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float2 v = row[ix[a]];
      rx = fmaf(wx[a], v.x, rx);
      ry = fmaf(wx[a], v.y, ry);
    }
    Ux = fmaf(wy[b], rx, Ux);
    Uy = fmaf(wy[b], ry, Uy);
  }
  return make_float2(Ux, Uy);
}

// The world's fluid velocity at bead position p.
__device__ __forceinline__ float2 interp_u(const WorldDev& w, const float4 p) { return interp_field(w.u, w.W, w.H, p); }

// ---------------------------------------------------------------------------
// Two-layer filament (Fluid-filament Interaction): the immersed-boundary
// points of bead i are X_i +- delta n_i.
// ---------------------------------------------------------------------------

__device__ __forceinline__ float2 layer_velocity(const WorldDev& w, const float4 p, float2 n, float d) {
  int cx, cy;
  float fx, fy;
  layer_cell(p, n, d, w.W, w.H, cx, cy, fx, fy);
  float wx[4], wy[4];
  peskin4(fx, wx);
  peskin4(fy, wy);
  float Ux = 0.0f, Uy = 0.0f;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const float2* row = w.u + (size_t)wrap_once(cy - 1 + b, w.H) * w.W;
    float rx = 0.0f, ry = 0.0f;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float2 v = row[wrap_once(cx - 1 + a, w.W)];
      rx = fmaf(wx[a], v.x, rx);
      ry = fmaf(wx[a], v.y, ry);
    }
    Ux = fmaf(wy[b], rx, Ux);
    Uy = fmaf(wy[b], ry, Uy);
  }
  return make_float2(Ux, Uy);
}

// The energy field sampled at p with the interpolation kernel.
__device__ __forceinline__ float energy_sample(const WorldDev& w, const float4 q) {
  const int W = w.W, H = w.H;
  float ex[4], ey[4];
  peskin4(q.x, ex);
  peskin4(q.y, ey);
  const int qx = cell_x(q), qy = cell_y(q);
  float e = 0.0f;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const float* row = w.energy + (size_t)wrap_once(qy - 1 + b, H) * W;
    float r = 0.0f;
#pragma unroll
    for (int a = 0; a < 4; ++a) r = fmaf(ex[a], row[wrap_once(qx - 1 + a, W)], r);
    e = fmaf(ey[b], r, e);
  }
  return e;
}

// a8's velocity of bead i at p = X^n: the interpolated fluid velocity, or,
// for a two-layer filament, the mean of the velocities at X +- delta n.
// With observables and an energy field (kExt), also the bead's energy
// sample at X^n, stored in ebead and added to q in fixed point.
// The energy bead i collects at p (observables with an energy field): stored
// in ebead and added to q in fixed point.
__device__ __forceinline__ void bead_energy(const WorldDev& w, int i, const float4 p, long long& q) {
  if (w.observe && w.energy) {
    const float e = energy_sample(w, p);
    w.ebead[i] = e;
    q += obs_q(e);
  }
}

// (the extended worlds' part: U is the velocity interpolated at p)
__device__ __forceinline__ float2 bead_velocity_ext(const WorldDev& w, int i, const float4 p, float2 U, long long& q) {
  bead_energy(w, i, p, q);
  if (w.layers == 2) {
    const float2 n = w.nrm[i];
    const float2 Up = layer_velocity(w, p, n, w.layer_half), Um = layer_velocity(w, p, n, -w.layer_half);
    return make_float2(0.5f * (Up.x + Um.x), 0.5f * (Up.y + Um.y));
  }
  return U;
}

template <bool kExt>
__device__ __forceinline__ float2 bead_velocity(const WorldDev& w, int i, const float4 p, long long& q) {
  float2 U = make_float2(0.0f, 0.0f);
  if (!(kExt && w.layers == 2)) U = interp_u(w, p);
  if (kExt) U = bead_velocity_ext(w, i, p, U, q);
  return U;
}

__device__ __forceinline__ float sq(float v) { return v * v; }

// Constants of the PBD passes, read once per warp.
struct PbdConst {
  float hb, hs, ksh, ko, kappa_dt, dt, u_max;
  int n_pbd, order, W, H, nbx;
};

__device__ __forceinline__ PbdConst pbd_const(const WorldDev& w) {
  PbdConst k;
  k.hb = 0.5f * w.k_bend;
  k.hs = 0.5f * w.k_st;
  k.ksh = w.k_sh;
  k.ko = w.orient * k.hs * k.ksh;
  k.kappa_dt = w.kappa_dt;
  k.dt = w.dt;
  k.u_max = w.u_max;
  k.n_pbd = w.n_pbd;
  k.order = w.pbd_order;
  k.W = w.W;
  k.H = w.H;
  k.nbx = w.nbx;
  return k;
}

// The per-edge factors of the position pass: sc = (l - L)/l = 1 - L/l with
// l = |(x, y)| (from the hardware reciprocal square root), and the sine and
// cosine of the frame angle (the hardware's, of the angle reduced to
// [-pi, pi]).  Their errors (a few 1e-7) stay below the step's float32
// resolution of the elastic force.
__device__ __forceinline__ void pbd_edge_terms(float x, float y, float L, float th, float& sc, float& sn, float& cs) {
  sc = fmaf(-L, rsqrtf(x * x + y * y), 1.0f);
  const float tr = fmaf(-6.28318548f, rintf(th * 0.159154943f), th);
  __sincosf(tr, &sn, &cs);
}

// Position pass of one edge (Eqs. 2-4) with current edge vector (x, y),
// rest length L (iL = 1 / L) and frame angle th: the correction (ddx, ddy) of
// its first bead (the second gets the opposite), and the frame's turn toward
// the edge.
__device__ __forceinline__ void edge_correction(float x, float y, float L, float iL, float& th, const PbdConst& k,
                                                float& ddx, float& ddy) {
  float sc, sn, cs;
  pbd_edge_terms(x, y, L, th, sc, sn, cs);
  const float csx = sc * x, csy = sc * y;
  ddx = k.hs * (csx + k.ksh * (x - L * cs - csx));
  ddy = k.hs * (csy + k.ksh * (y - L * sn - csy));
  th += k.ko * (cs * y - sn * x) * iL;   // frame turns toward the edge (orient)
}

// Unit normal of the filament at a bead (two-layer coupling): t is the
// normalised sum of the unit vectors of the bead's outgoing and incoming
// edges; where they nearly cancel (|sum| < 1e-3, a chain folded back) t is
// the outgoing edge, the incoming one at the last bead; n = (-t_y, t_x).
__device__ __forceinline__ float2 unit2(float2 v) {
  const float r = rsqrtf(v.x * v.x + v.y * v.y);
  return make_float2(v.x * r, v.y * r);
}

__device__ __forceinline__ float2 bead_normal(float2 out, bool has_out, float2 in, bool has_in) {
  float sx = 0.0f, sy = 0.0f;
  if (has_out) {
    sx += out.x;
    sy += out.y;
  }
  if (has_in) {
    sx += in.x;
    sy += in.y;
  }
  const float ns = sqrtf(sx * sx + sy * sy);
  float2 t;
  if (ns >= 1e-3f) t = make_float2(sx / ns, sy / ns);
  else t = has_out ? out : in;
  return make_float2(-t.y, t.x);
}

// a2: lanes of one warp that share a bin take consecutive places from one
// atomic on its count.  bin_claim starts it (valid lanes pass their bin,
// the others a negative one of their own); bin_place returns the lane's slot.
// Every lane calls both; two claims can be in flight before their places.
struct BinClaim {
  int base, lo, hi;   // the group's first place; the bin's slots
  unsigned peers;
};

__device__ __forceinline__ BinClaim bin_claim(const WorldDev& w, int* counts, bool valid, int bin) {
  const int lane = threadIdx.x & 31;
  BinClaim c;
  c.peers = __match_any_sync(0xffffffffu, valid ? bin : -1 - lane);
  c.base = c.lo = c.hi = 0;
  if (valid) {
    c.lo = w.bin_base[bin];
    c.hi = w.bin_base[bin + 1];
  }
  if (valid && (__ffs(c.peers) - 1) == lane) c.base = atomicAdd(&counts[bin], __popc(c.peers));
  return c;
}

__device__ __forceinline__ int bin_place(const WorldDev& w, int* counts, bool valid, const BinClaim& c) {
  const int lane = threadIdx.x & 31;
  const int at = __shfl_sync(0xffffffffu, c.base, __ffs(c.peers) - 1) + __popc(c.peers & ((1u << lane) - 1u));
  if (!valid) return -1;
  if (c.lo + at < c.hi) return c.lo + at;
  // the bin's slots are full (never more beads than N, unless a run that timed
  // out left counts behind)
  return w.slot_end + min(atomicAdd(&counts[w.n_bins], 1), w.N - 1);
}

// The bin of the bead at P.
__device__ __forceinline__ int bead_bin_of(const float4& P, int nbx) {
  return (cell_y(P) / kBin) * nbx + cell_x(P) / kBin;
}

// The bead's record in its slot, and the slot by bead where a later kernel
// asks for it.
__device__ __forceinline__ void bin_store(const WorldDev& w, int slot, int b, const float4& P, float2 fe) {
  w.bpos[slot] = P;
  w.brec[slot] = make_float4(fe.x, fe.y, __int_as_float(b), 0.0f);
  if (w.bead_slot) w.bead_slot[b] = slot;
}

// With direct forcing the PBD's output for a bead is its velocity U_s =
// U* + dl/dt, U* (the fluid's, stored in ubead by the prediction) plus the
// PBD correction of the carried position.
__device__ __forceinline__ void bead_out_velocity(const WorldDev& w, const PbdConst& k, int b, float dlx, float dly) {
  const float2 U = w.ubead[b];
  const float2 Us = make_float2(U.x + dlx / k.dt, U.y + dly / k.dt);
  w.ubead[b] = Us;
  w.sus[w.bead_slot[b]] = Us;   // the MDF passes read U_s by slot
}

// F_el = kappa (x_hat - X) / dt of one bead; with `fields`, kept with its
// bin for read-out.
__device__ __forceinline__ float2 bead_out_force(const WorldDev& w, const PbdConst& k, int b, int bin, float dlx,
                                                 float dly, int fields, float& fmax) {
  const float2 fe = make_float2(k.kappa_dt * dlx, k.kappa_dt * dly);
  fmax = fmaxf(fmax, fmaxf(fabsf(fe.x), fabsf(fe.y)));
  if (fields) {
    w.fel[b] = fe;
    w.bead_bin[b] = bin;
  }
  return fe;
}

// Jacobi PBD of a filament of at most 64 beads in registers: lane l holds
// beads, edges and joints 2l and 2l + 1, and reads its neighbours' values by
// warp shuffles.  The same arithmetic, in the same order, as pbd_block.
// kEarly: the beads claim their places in the bins, which depend on the
// positions alone, before the passes, so that the atomics' round trip
// overlaps them (a warp alone on its scheduler waited some 2,300 cycles of
// 10,500 for them; with many warps the registers it holds cost more).
template <bool kExt, int kMode, bool kEarly>
__device__ __forceinline__ float pbd_regs(const WorldDev& w, const PbdConst& k, int b0, int B, int e0, int j0,
                                          long long t, int fields) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int nE = B - 1, nJ = B - 2;
  const int i0 = 2 * lane, i1 = i0 + 1;
  const bool hb0 = i0 < B, hb1 = i1 < B, he0 = i0 < nE, he1 = i1 < nE, hj0 = i0 < nJ, hj1 = i1 < nJ;
  const float4 z4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  // every load that needs only the work item first, then (kMode 1, 2) the
  // gathers of both beads before either's arithmetic: a step of a small world
  // is a chain of memory round trips of some 0.4 us each
  float4 P0 = hb0 ? w.pos[b0 + i0] : z4;
  float4 P1 = hb1 ? w.pos[b0 + i1] : z4;
  float2 D0 = make_float2(0.0f, 0.0f), D1 = D0;
  if (kMode == 1) {
    if (hb0) D0 = w.disp[b0 + i0];
    if (hb1) D1 = w.disp[b0 + i1];
  }
  float th0 = he0 ? w.theta[e0 + i0] : 0.0f;
  float th1 = he1 ? w.theta[e0 + i1] : 0.0f;
  const float L0 = he0 ? (kExt ? rest_length(w, e0 + i0, t) : w.L_rest[e0 + i0]) : 1.0f;
  const float L1 = he1 ? (kExt ? rest_length(w, e0 + i1, t) : w.L_rest[e0 + i1]) : 1.0f;
  const float4 dr0 = hj0 ? w.drive[j0 + i0] : z4, dr1 = hj1 ? w.drive[j0 + i1] : z4;
  const float iL0 = __frcp_rn(L0), iL1 = __frcp_rn(L1);
  float2 U0 = make_float2(0.0f, 0.0f), U1 = U0;
  if (kMode == 1 && !(kExt && w.layers == 2)) {
    // (lanes without a bead gather at cell 0: valid, unused)
    U0 = interp_u(w, P0);
    U1 = interp_u(w, P1);
  } else if (kMode == 2) {
    const float2* u = mdf_u(w, 0);   // u*
    U0 = interp_field(u, w.W, w.H, P0);
    U1 = interp_field(u, w.W, w.H, P1);
  }
  const float thr0 = hj0 ? drive_angle(dr0, t) : 0.0f;
  const float thr1 = hj1 ? drive_angle(dr1, t) : 0.0f;
  if (kMode == 1) {
    // a8 of the previous step for the lane's beads, then this step's PBD from X^n
    long long q = 0;
    if (kExt) {
      if (hb0) U0 = bead_velocity_ext(w, b0 + i0, P0, U0, q);
      if (hb1) U1 = bead_velocity_ext(w, b0 + i1, P1, U1, q);
    }
    if (hb0) P0 = advance_tail<false>(w, k.u_max, b0 + i0, P0, D0, U0.x, U0.y);
    if (hb1) P1 = advance_tail<false>(w, k.u_max, b0 + i1, P1, D1, U1.x, U1.y);
    if (kExt && w.observe && w.energy) obs_add_warp(&w.obs[2], q);
  } else if (kMode == 0 && w.rec_pos) {
    // the step's start, into the reverse mode's record
    if (hb0) w.rec_pos[b0 + i0] = P0;
    if (hb1) w.rec_pos[b0 + i1] = P1;
    if (he0) w.rec_theta[e0 + i0] = th0;
    if (he1) w.rec_theta[e0 + i1] = th1;
  } else if (kMode == 2) {
    // direct forcing: the fluid (u*) carries the beads, PBD starts there
    if (hb0) {
      w.ubead[b0 + i0] = U0;
      P0 = advance_pos(w, P0, U0.x, U0.y);
    }
    if (hb1) {
      w.ubead[b0 + i1] = U1;
      P1 = advance_pos(w, P1, U1.x, U1.y);
    }
  }
  float4 Pn;   // bead 2l + 2
  Pn.x = __shfl_down_sync(kAll, P0.x, 1);
  Pn.y = __shfl_down_sync(kAll, P0.y, 1);
  Pn.z = __shfl_down_sync(kAll, P0.z, 1);
  Pn.w = __shfl_down_sync(kAll, P0.w, 1);
  const float2 v0 = edge_vec(P0, P1, k.W, k.H);
  const float2 v1 = edge_vec(P1, Pn, k.W, k.H);
  if (kExt && w.layers == 2) {
    // filament normals at beads 2l, 2l + 1 from X^n
    const float2 z2 = make_float2(0.0f, 0.0f);
    const float2 u0 = he0 ? unit2(v0) : z2, u1 = he1 ? unit2(v1) : z2;
    float2 um;   // edge 2l - 1, incoming at bead 2l
    um.x = __shfl_up_sync(kAll, u1.x, 1);
    um.y = __shfl_up_sync(kAll, u1.y, 1);
    if (hb0) w.nrm[b0 + i0] = bead_normal(u0, he0, um, lane > 0);
    if (hb1) w.nrm[b0 + i1] = bead_normal(u1, he1, u0, true);
  }
  int* counts = nullptr;
  BinClaim c0, c1;
  if (kMode != 2 && kEarly) {
    counts = step_counts(w, t);
    c0 = bin_claim(w, counts, hb0, bead_bin_of(P0, k.nbx));
    c1 = bin_claim(w, counts, hb1, bead_bin_of(P1, k.nbx));
  }
  float dlx0 = 0.0f, dly0 = 0.0f, dlx1 = 0.0f, dly1 = 0.0f;
  if (k.order == 1) {
    for (int iter = 0; iter < k.n_pbd; ++iter) {
      // bending pass (Eq. 1), joint 2l of every lane first, then joint 2l + 1
      // from the updated angles: joint j moves theta_j by +h C_j and
      // theta_{j+1} by -h C_j
      const float C0 = hj0 ? th1 - th0 - thr0 : 0.0f;
      if (hj0) {
        th0 += k.hb * C0;
        th1 -= k.hb * C0;
      }
      const float thn = __shfl_down_sync(kAll, th0, 1);   // theta_{2l+2}, updated
      const float C1 = hj1 ? thn - th1 - thr1 : 0.0f;
      if (hj1) th1 += k.hb * C1;
      const float Cm = __shfl_up_sync(kAll, C1, 1);        // joint 2l-1 moves theta_{2l}
      if (lane > 0) th0 -= k.hb * Cm;
      // position pass (Eqs. 2-4), edge 2l first, then edge 2l + 1
      float ddx0 = 0.0f, ddy0 = 0.0f;
      if (he0) {
        edge_correction(v0.x + (dlx1 - dlx0), v0.y + (dly1 - dly0), L0, iL0, th0, k, ddx0, ddy0);
        dlx0 += ddx0;
        dly0 += ddy0;
        dlx1 -= ddx0;
        dly1 -= ddy0;
      }
      const float dlxn = __shfl_down_sync(kAll, dlx0, 1), dlyn = __shfl_down_sync(kAll, dly0, 1);
      float ddx1 = 0.0f, ddy1 = 0.0f;
      if (he1) {
        edge_correction(v1.x + (dlxn - dlx1), v1.y + (dlyn - dly1), L1, iL1, th1, k, ddx1, ddy1);
        dlx1 += ddx1;
        dly1 += ddy1;
      }
      const float ddxm = __shfl_up_sync(kAll, ddx1, 1), ddym = __shfl_up_sync(kAll, ddy1, 1);
      if (lane > 0) {   // edge 2l-1 moves bead 2l (its second bead)
        dlx0 -= ddxm;
        dly0 -= ddym;
      }
    }
  }
  for (int iter = 0; iter < (k.order == 1 ? 0 : k.n_pbd); ++iter) {
    // bending pass (Eq. 1): C_j = (theta_{j+1} - theta_j) - theta_rest,j
    const float thn = __shfl_down_sync(kAll, th0, 1);
    const float C0 = hj0 ? th1 - th0 - thr0 : 0.0f;
    const float C1 = hj1 ? thn - th1 - thr1 : 0.0f;
    const float Cm = __shfl_up_sync(kAll, C1, 1);   // C_{2l-1}
    if (he0) th0 += k.hb * (C0 - (lane > 0 ? Cm : 0.0f));
    if (he1) th1 += k.hb * (C1 - C0);
    // position pass (Eqs. 2-4) on the updated frames
    const float dlxn = __shfl_down_sync(kAll, dlx0, 1), dlyn = __shfl_down_sync(kAll, dly0, 1);
    float ddx0 = 0.0f, ddy0 = 0.0f, ddx1 = 0.0f, ddy1 = 0.0f;
    if (he0) edge_correction(v0.x + (dlx1 - dlx0), v0.y + (dly1 - dly0), L0, iL0, th0, k, ddx0, ddy0);
    if (he1) edge_correction(v1.x + (dlxn - dlx1), v1.y + (dlyn - dly1), L1, iL1, th1, k, ddx1, ddy1);
    const float ddxm = __shfl_up_sync(kAll, ddx1, 1), ddym = __shfl_up_sync(kAll, ddy1, 1);
    if (hb0) {
      dlx0 += ddx0 - (lane > 0 ? ddxm : 0.0f);
      dly0 += ddy0 - (lane > 0 ? ddym : 0.0f);
    }
    if (hb1) {
      dlx1 += ddx1 - ddx0;
      dly1 += ddy1 - ddy0;
    }
  }
  if (he0) w.theta[e0 + i0] = th0;
  if (he1) w.theta[e0 + i1] = th1;
  float fmax = 0.0f;
  if (kMode == 2) {
    if (hb0) bead_out_velocity(w, k, b0 + i0, dlx0, dly0);
    if (hb1) bead_out_velocity(w, k, b0 + i1, dlx1, dly1);
  } else {
    const int bin0 = bead_bin_of(P0, k.nbx), bin1 = bead_bin_of(P1, k.nbx);
    float2 fe0 = make_float2(0.0f, 0.0f), fe1 = fe0;
    if (hb0) fe0 = bead_out_force(w, k, b0 + i0, bin0, dlx0, dly0, fields, fmax);
    if (hb1) fe1 = bead_out_force(w, k, b0 + i1, bin1, dlx1, dly1, fields, fmax);
    if (!kEarly) {
      counts = step_counts(w, t);
      c0 = bin_claim(w, counts, hb0, bin0);
      c1 = bin_claim(w, counts, hb1, bin1);
    }
    const int s0 = bin_place(w, counts, hb0, c0), s1 = bin_place(w, counts, hb1, c1);
    if (hb0) bin_store(w, s0, b0 + i0, P0, fe0);
    if (hb1) bin_store(w, s1, b0 + i1, P1, fe1);
  }
  if (kExt && w.observe && t >= 1) {
    // behaviour descriptors (Eqs. 5, 6): squared change of the rest angles
    // and rest lengths from step t - 1 to step t
    float eb = 0.0f, ep = 0.0f;
    if (hj0) eb += sq(drive_angle(w.drive[j0 + i0], t - 1) - thr0);
    if (hj1) eb += sq(drive_angle(w.drive[j0 + i1], t - 1) - thr1);
    if (w.ldrive) {
      if (he0) ep += sq(rest_length(w, e0 + i0, t - 1) - L0);
      if (he1) ep += sq(rest_length(w, e0 + i1, t - 1) - L1);
    }
    obs_add_warp(&w.obs[0], obs_q(eb));
    obs_add_warp(&w.obs[1], obs_q(ep));
  }
  return fmax;
}

// PBD of a filament of more than 64 beads by one block: the filament's
// edges, joints and bead corrections live in shared memory; every pass reads
// them, then writes corrections, with a block barrier in between, so all
// corrections of a pass see the state before it.  A pass over a long chain
// is bound by the latency of its rounds: with one warp a filament of 300
// beads took ten rounds a pass, and the fused advance + PBD of 60 filaments
// of 2 to 300 beads 33.7 us; with a block 11.0 us.
template <bool kExt, int kMode>
__device__ __forceinline__ float pbd_block(const WorldDev& w, const PbdConst& k, int b0, int B, int e0, int j0,
                                          long long t, int fields, float* s, int maxB) {
  const int tid = threadIdx.x, T = blockDim.x;
  const int nE = B - 1, nJ = B - 2;
  float* vx = s;
  float* vy = s + maxB;
  float* th = s + 2 * maxB;
  float* Lr = s + 3 * maxB;
  float* ddx = s + 4 * maxB;
  float* ddy = s + 5 * maxB;
  float* dlx = s + 6 * maxB;
  float* dly = s + 7 * maxB;
  float* thr = s + 8 * maxB;
  float* C = s + 9 * maxB;
  float4* P = reinterpret_cast<float4*>(s + 10 * maxB);    // bead positions
  float4* D = reinterpret_cast<float4*>(s + 14 * maxB);    // joint drive parameters
  // stage the filament's inputs in shared memory, every copy in flight at once
  if (kMode == 1) {
    // a8 of the previous step, the advanced positions staged directly
    long long q = 0;
    for (int i = tid; i < B; i += T) {
      const float4 p = w.pos[b0 + i];
      const float2 d = w.disp[b0 + i];
      const float2 U = bead_velocity<kExt>(w, b0 + i, p, q);
      P[i] = advance_tail<false>(w, k.u_max, b0 + i, p, d, U.x, U.y);
    }
    if (kExt && w.observe && w.energy) obs_add_warp(&w.obs[2], q);
  } else if (kMode == 2) {
    // direct forcing: the positions the fluid (u*) carries the beads to
    for (int i = tid; i < B; i += T) {
      const float4 p = w.pos[b0 + i];
      const float2 U = interp_field(mdf_u(w, 0), w.W, w.H, p);
      w.ubead[b0 + i] = U;
      P[i] = advance_pos(w, p, U.x, U.y);
    }
  } else {
    for (int i = tid; i < B; i += T) cpa16(&P[i], &w.pos[b0 + i]);
  }
  for (int e = tid; e < nE; e += T) {
    cpa4(&th[e], &w.theta[e0 + e]);
    if (!kExt || !w.ldrive) cpa4(&Lr[e], &w.L_rest[e0 + e]);
    else Lr[e] = drive_length(w.ldrive[e0 + e], t);
  }
  for (int j = tid; j < nJ; j += T) cpa16(&D[j], &w.drive[j0 + j]);
  cpa_wait_all();
  __syncthreads();
  if (kMode == 0 && w.rec_pos) {   // the step's start, into the reverse mode's record
    for (int i = tid; i < B; i += T) w.rec_pos[b0 + i] = P[i];
    for (int e = tid; e < nE; e += T) w.rec_theta[e0 + e] = th[e];
  }
  for (int e = tid; e < nE; e += T) {
    const float2 v = edge_vec(P[e], P[e + 1], k.W, k.H);
    vx[e] = v.x;
    vy[e] = v.y;
  }
  for (int j = tid; j < nJ; j += T) thr[j] = drive_angle(D[j], t);
  for (int i = tid; i < B; i += T) {
    dlx[i] = 0.0f;
    dly[i] = 0.0f;
  }
  __syncthreads();
  if (kExt && w.layers == 2) {
    for (int i = tid; i < B; i += T) {
      const float2 z2 = make_float2(0.0f, 0.0f);
      const float2 out = i < nE ? unit2(make_float2(vx[i], vy[i])) : z2;
      const float2 in = i > 0 ? unit2(make_float2(vx[i - 1], vy[i - 1])) : z2;
      w.nrm[b0 + i] = bead_normal(out, i < nE, in, i > 0);
    }
  }
  if (k.order == 1) {
    // red-black passes: within a colour no two joints share an edge and no
    // two edges share a bead, so the lanes update in place
    for (int iter = 0; iter < k.n_pbd; ++iter) {
      for (int c = 0; c < 2; ++c) {
        for (int j = 2 * tid + c; j < nJ; j += 2 * T) {
          const float Cj = th[j + 1] - th[j] - thr[j];
          th[j] += k.hb * Cj;
          th[j + 1] -= k.hb * Cj;
        }
        __syncthreads();
      }
      for (int c = 0; c < 2; ++c) {
        for (int e = 2 * tid + c; e < nE; e += 2 * T) {
          float the = th[e], ddxe, ddye;
          edge_correction(vx[e] + (dlx[e + 1] - dlx[e]), vy[e] + (dly[e + 1] - dly[e]), Lr[e], __frcp_rn(Lr[e]), the, k, ddxe, ddye);
          th[e] = the;
          dlx[e] += ddxe;
          dly[e] += ddye;
          dlx[e + 1] -= ddxe;
          dly[e + 1] -= ddye;
        }
        __syncthreads();
      }
    }
  }
  for (int iter = 0; iter < (k.order == 1 ? 0 : k.n_pbd); ++iter) {
    for (int j = tid; j < nJ; j += T) C[j] = th[j + 1] - th[j] - thr[j];
    __syncthreads();
    for (int e = tid; e < nE; e += T) {
      const float c1 = e < nJ ? C[e] : 0.0f;      // edge e is theta_1 of joint e
      const float c0 = e > 0 ? C[e - 1] : 0.0f;   // ... and theta_2 of joint e-1
      th[e] += k.hb * (c1 - c0);
    }
    __syncthreads();
    for (int e = tid; e < nE; e += T) {
      float the = th[e];
      edge_correction(vx[e] + (dlx[e + 1] - dlx[e]), vy[e] + (dly[e + 1] - dly[e]), Lr[e], __frcp_rn(Lr[e]), the, k, ddx[e], ddy[e]);
      th[e] = the;
    }
    __syncthreads();
    for (int i = tid; i < B; i += T) {
      const float ax = i < nE ? ddx[i] : 0.0f, ay = i < nE ? ddy[i] : 0.0f;          // x_1 of edge i
      const float bx = i > 0 ? ddx[i - 1] : 0.0f, by = i > 0 ? ddy[i - 1] : 0.0f;    // x_2 of edge i-1
      dlx[i] += ax - bx;
      dly[i] += ay - by;
    }
    __syncthreads();
  }
  for (int e = tid; e < nE; e += T) w.theta[e0 + e] = th[e];
  float fmax = 0.0f;
  if (kMode == 2) {
    for (int i = tid; i < B; i += T) bead_out_velocity(w, k, b0 + i, dlx[i], dly[i]);
  } else {
    int* counts = step_counts(w, t);
    for (int i0 = 0; i0 < B; i0 += T) {
      const int i = i0 + tid;
      const bool valid = i < B;
      const float4 p = valid ? P[i] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      const int bin = bead_bin_of(p, k.nbx);
      const BinClaim c = bin_claim(w, counts, valid, bin);
      float2 fe = make_float2(0.0f, 0.0f);
      if (valid) fe = bead_out_force(w, k, b0 + i, bin, dlx[i], dly[i], fields, fmax);
      const int slot = bin_place(w, counts, valid, c);
      if (valid) bin_store(w, slot, b0 + i, p, fe);
    }
  }
  if (kExt && w.observe && t >= 1 && tid < 32) {
    // the first warp alone, so that the rounding of its partial sums does not
    // depend on the width of the block
    float eb = 0.0f, ep = 0.0f;
    for (int j = tid; j < nJ; j += 32) eb += sq(drive_angle(D[j], t - 1) - thr[j]);
    if (w.ldrive)
      for (int e = tid; e < nE; e += 32) ep += sq(drive_length(w.ldrive[e0 + e], t - 1) - Lr[e]);
    obs_add_warp(&w.obs[0], obs_q(eb));
    obs_add_warp(&w.obs[1], obs_q(ep));
  }
  return fmax;
}

// a1 + a3 + a2 of the filaments of a launch: its list holds the n_long of
// more than 64 beads first, one block each (pbd_block), then the others, one
// warp each in registers, wpb to a block.  Bead positions enter as edge
// vectors v0 = min_image(X_b - X_a) plus the accumulated corrections, so the
// corrections keep full FP32 precision whatever the magnitude of the
// coordinates.
struct PbdWork {
  int n_long, n_items;   // filaments of more than 64 beads, all filaments
  int wpb;               // filaments a block of the others takes
  int maxB;              // slots per array of the block's dynamic shared memory (a multiple of 4: float4 arrays stay aligned)
};
extern __shared__ __align__(16) float pbd_dyn_smem[];

// kLong: the launch has such filaments (a kernel of its own: holding both
// forms costs the warp form registers, 150 -> 167 us at 2^22 beads).
template <bool kExt, int kMode, bool kSingle, bool kLong, bool kEarly>
__device__ __forceinline__ void pbd_body(const WorldDev* __restrict__ worlds, const int4* __restrict__ items,
                                         const PbdWork& pw, int off, int fields, unsigned blk) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_long = kLong ? pw.n_long : 0;
  const bool is_long = kLong && (int)blk < n_long;   // block-uniform
  const int item = is_long ? (int)blk : n_long + ((int)blk - n_long) * pw.wpb + warp;
  if (!is_long && (warp >= pw.wpb || item >= pw.n_items)) return;  // warp-uniform exit; no block barrier follows
  const int4 it = items[item];
  // (a single-world launch's descriptor need not wait for the item)
  const WorldDev& w = worlds[kSingle ? 0 : it.x];
  if ((kMode == 2) != (w.ib == 1)) return;   // direct-forcing worlds run their PBD after the steric spread
  const int f = it.y, b0 = it.z, B = it.w;
  const int e0 = b0 - f, j0 = b0 - 2 * f;
  const long long t = *w.t + off;
  const PbdConst k = pbd_const(w);
  float fmax;
  if (kLong && is_long) fmax = pbd_block<kExt, kMode>(w, k, b0, B, e0, j0, t, fields, pbd_dyn_smem, pw.maxB);
  else fmax = pbd_regs<kExt, kMode, kEarly>(w, k, b0, B, e0, j0, t, fields);
  if (kMode == 2) return;
  // largest |F_el| component of the world this step (bounds the spread's
  // fixed-point scale); non-negative floats order like their bit patterns
  for (int o = 16; o > 0; o >>= 1) fmax = fmaxf(fmax, __shfl_xor_sync(0xffffffffu, fmax, o));
  if (lane == 0) atomicMax(&w.fel_max[t & 1], __float_as_uint(fmax));
}

// a8: U_i = sum_c delta_h(c - X_i) u(c) over the 4x4 stencil, then the
// inertia-free advance X += dt U (cell index + fraction, wrapped) and the
// unwrapped displacement D += dt U.  Thread 0 of each world's first block
// advances the world's step counter by the inc steps of the run that this
// advance ends (no other thread of the launch reads it).
template <bool kExt, bool kSingle>
__device__ __forceinline__ void interp_advance_body(const WorldDev* __restrict__ worlds,
                                                    const int2* __restrict__ items, int inc, unsigned blk) {
  const int2 it = kSingle ? make_int2(0, (int)blk * kBeadChunk) : items[blk];
  const WorldDev& w = worlds[it.x];
  if (it.y == 0 && threadIdx.x == 0) *w.t += inc;
  const int i = it.y + threadIdx.x;
  // the velocity at the bead's position at the start of the step (and, with
  // observables, the energy sampled there; every lane of the block takes
  // part in the warp sum)
  long long q = 0;
  float4 p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float2 U = make_float2(0.0f, 0.0f);
  float2 d = make_float2(0.0f, 0.0f);
  const float u_max = w.u_max;
  if (i < w.N) {
    p = w.pos[i];
    d = w.disp[i];
    if (kExt && w.ib == 1) {
      U = w.ubead[i];   // direct forcing: the bead's own velocity U_s
      bead_energy(w, i, p, q);
    } else {
      U = bead_velocity<kExt>(w, i, p, q);
    }
  }
  if (kExt && w.observe && w.energy) obs_add_warp(&w.obs[2], q);
  if (i >= w.N) return;
  advance_tail(w, u_max, i, p, d, U.x, U.y);
}

}  // namespace mc
