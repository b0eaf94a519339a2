// The first part of a step: predictor and wrap, cell key, histogram.  Run by
// the sort's first kernel, or, inside a run of steps, by the corrector of the
// step before (k_gather<NEXT>), which has the velocities and accelerations in
// registers.
#pragma once

#include "dss_internal.cuh"

// What the sort's first kernel writes.
struct SortOut {
  int* key;                 // cell of each particle (source order)
  int* cell_count;          // histogram of the keys (cleared behind the scan)
  int* tile_count;          // its sums over the scan's tiles (null: too many)
  int* cell_ids;            // per cell a row of bcap ids
  int bcap;
  // ids beyond a cell's row: a chain of links per cell, each the particles that
  // one warp brought (a mask of its lanes), kept at the first one's index.
  // Consecutive particles are neighbours in space, so that a link holds many of
  // the cell; no cell's fullness costs memory or work elsewhere.
  int* more;                // per cell: index + 1 of its last link (cleared by the row pass)
  int* link_next;
  unsigned* link_lanes;
  double* pred;             // 6n: predicted position and velocity
  signed char* xc;          // y crossings
  unsigned long long* scan_status;   // the look-back state of the cell scan
  int* scan_ticket;
  int scan_words;
  int* row_sums;                     // and the row sums of its search
  int row_words;
  StepGeo* sg;
};

inline SortOut sort_out(const dss_handle* h) {
  return SortOut{h->key,
                 h->cell_count,
                 scan_tiles_for(h->g.ncell) <= kScanTiles ? h->tile_count : nullptr,
                 h->cell_ids,
                 h->cell_cap,
                 h->cell_more,
                 h->tmp,
                 reinterpret_cast<unsigned*>(h->offs),
                 h->pred,
                 h->xc,
                 h->scan_status,
                 h->scan_ticket,
                 h->scan_tiles_max,
                 h->row_sums,
                 h->row_words,
                 h->sg};
}

// Predictor of Eq. 15a-b and the wrap of Eq. 16 for one particle; computed
// once per step and stored for the gather.  In FP64 mode each product and
// sum is rounded separately (the trajectory then differs from a plain FP64
// evaluation only through the order of the force sums); in mixed precision
// as fused multiply-adds (GB300's narrow FP64 pipe bounds this kernel).
// Returns the y crossing (-1 out through the top, +1 bottom).
// Comparisons for the wrap on the IEEE bit patterns (integer instructions
// instead of GB300's narrow FP64 pipe).  For L > 0 and any finite v the
// signed 64-bit order of the patterns is the order of the values on the
// non-negative side, and every negative v sorts below; -0.0 is not below 0.
__device__ __forceinline__ bool ge_pos(double v, double L) {
  return __double_as_longlong(v) >= __double_as_longlong(L);
}
__device__ __forceinline__ bool lt_zero(double v) {
  const long long b = __double_as_longlong(v);
  return b < 0 && b != (long long)0x8000000000000000ull;
}

struct Pred {
  double x, y, z, ux, uy, uz;
  int cross;
};

// Lees-Edwards wrap of Eq. 16 and the periodic wraps along x and z, for a
// particle that left the box (out of line: see f32_rn_slow).
static __device__ __noinline__ Pred wrap_out(const Geo& g, const InstGeo& I, const DevStatus* st, int adv, Pred r) {
  double x = r.x, y = r.y, z = r.z, ux = r.ux;
  // leaving through y >= L_y re-enters at the bottom shifted by -off along
  // x with u_x - gdot L_y, and vice versa
  const double Ly = I.L[1];
  if (ge_pos(y, Ly)) {
    y = __dsub_rn(y, Ly);
    x = __dsub_rn(x, le_offset(g, I, dev_nstep(st) + adv));
    r.cross = -1;
  } else if (lt_zero(y)) {
    y = __dadd_rn(y, Ly);
    x = __dadd_rn(x, le_offset(g, I, dev_nstep(st) + adv));
    r.cross = 1;
    if (ge_pos(y, Ly)) y = 0.0;
  }
  // x back into [0, L_x): two conditional shifts give the same bits as
  // fmod followed by the two corrections, for |x| < 2 L_x
  const double Lx = I.L[0];
  if (lt_zero(x)) x = __dadd_rn(x, Lx); else if (ge_pos(x, Lx)) x = __dsub_rn(x, Lx);
  if (lt_zero(x)) x = __dadd_rn(x, Lx); else if (ge_pos(x, Lx)) x = __dsub_rn(x, Lx);
  if (ge_pos(z, I.L[2])) {
    z = __dsub_rn(z, I.L[2]);
  } else if (lt_zero(z)) {
    z = __dadd_rn(z, I.L[2]);
    if (ge_pos(z, I.L[2])) z = 0.0;
  }
  if (r.cross != 0)
    ux = __dadd_rn(ux, __dmul_rn(__dmul_rn((double)r.cross, I.gdot), Ly));
  r.x = x; r.y = y; r.z = z; r.ux = ux;
  return r;
}

// Position (x, y, z), velocity u and linear acceleration al at a step's start
// -> the predicted position and velocity, wrapped (adv: the step's end, in
// steps after the status' count).
__device__ __forceinline__ Pred predict_one(const Geo& g, const InstGeo& I, const DevStatus* st, int adv, double x,
                                            double y, double z, double ux, double uy, double uz, double ax,
                                            double ay, double az) {
  Pred r;
  r.cross = 0;
  const double dt = g.dt;
  const double hdt2 = g.hdt2;
  const double hdt = g.hdt;
  if (g.precision == DSS_FP64) {
    // FP64 mode: every product and sum rounded on its own, in the order
    // x + dt u + (dt/2 dt) alpha of Eq. 15a (no contraction)
    r.x = __dadd_rn(__dadd_rn(x, __dmul_rn(dt, ux)), __dmul_rn(hdt2, ax));
    r.y = __dadd_rn(__dadd_rn(y, __dmul_rn(dt, uy)), __dmul_rn(hdt2, ay));
    r.z = __dadd_rn(__dadd_rn(z, __dmul_rn(dt, uz)), __dmul_rn(hdt2, az));
    r.ux = __dadd_rn(ux, __dmul_rn(hdt, ax));
    r.uy = __dadd_rn(uy, __dmul_rn(hdt, ay));
    r.uz = __dadd_rn(uz, __dmul_rn(hdt, az));
  } else {
    r.x = __fma_rn(hdt2, ax, __fma_rn(dt, ux, x));
    r.y = __fma_rn(hdt2, ay, __fma_rn(dt, uy, y));
    r.z = __fma_rn(hdt2, az, __fma_rn(dt, uz, z));
    r.ux = __fma_rn(hdt, ax, ux);
    r.uy = __fma_rn(hdt, ay, uy);
    r.uz = __fma_rn(hdt, az, uz);
  }
  // inside the box (nearly every particle): nothing to wrap
  if (ge_pos(r.y, I.L[1]) || lt_zero(r.y) || ge_pos(r.x, I.L[0]) || lt_zero(r.x) || ge_pos(r.z, I.L[2]) ||
      lt_zero(r.z))
    r = wrap_out(g, I, st, adv, r);
  return r;
}

// Cell coordinate floor(x / cs) along one axis, clamped to the grid (the
// FP64 product's floor, mostly decided in FP32: floor_mul).
__device__ __forceinline__ int cell_coord_fast(double v, double inv, float invf, int nc) {
  const int k = floor_mul(v, inv, invf);
  return k < 0 ? 0 : (k >= nc ? nc - 1 : k);
}

// Bin of a particle: its instance's bins, its size class's layer, its cell.
__device__ __forceinline__ int cell_key(const InstGeo& I, int cls, double x, double y, double z) {
  int cx = cell_coord_fast(x, I.inv_cs[0], I.inv_csf[0], I.nc[0]);
  int cy = cell_coord_fast(y, I.inv_cs[1], I.inv_csf[1], I.nc[1]);
  int cz = cell_coord_fast(z, I.inv_cs[2], I.inv_csf[2], I.nc[2]);
  return I.cell_base + cls * I.ncell_layer + (cz * I.nc[1] + cy) * I.nc[0] + cx;
}

// The particle's key, its count and its id in the cell's row, or in a link of the
// cell's chain (called by all active lanes of a warp together; i lies at the
// lane's place in a row of 32).
__device__ __forceinline__ void key_insert(const SortOut& q, int i, int k, int id) {
  const unsigned act = __activemask();
  const unsigned peers = __match_any_sync(act, k);
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(peers) - 1;
  const int rank = __popc(peers & ((1u << lane) - 1u));
  int base = 0;
  if (lane == leader) base = atomicAdd(&q.cell_count[k], __popc(peers));
  if (q.tile_count) {
    // mostly one tile a warp: neighbours in memory are neighbours in space, and
    // for that the sums are kept in copies (one copy: 1M 32 -> 47 us)
    const int t = k / kScanTile;
    int one;
    int* const tc = q.tile_count + (blockIdx.x % kTileCopies) * kScanTiles;
    __match_all_sync(act, t, &one);
    if (one) {
      if (lane == __ffs(act) - 1) atomicAdd(&tc[t], __popc(act));
    } else if (lane == leader) {
      atomicAdd(&tc[t], __popc(peers));
    }
  }
  base = __shfl_sync(peers, base, leader) + rank;
  q.key[i] = k;
  if (base < q.bcap) {
    q.cell_ids[(int64_t)k * q.bcap + base] = id;
  } else if (base == q.bcap || rank == 0) {   // the first of the warp's beyond the row
    q.link_lanes[i] = peers & (0xffffffffu << lane);
    q.link_next[i] = atomicExch(&q.more[k], i + 1);
  }
}

__device__ __forceinline__ void store_pred(const SortOut& q, int n, int i, const Pred& p) {
  q.pred[i] = p.x;
  q.pred[n + i] = p.y;
  q.pred[2 * n + i] = p.z;
  q.pred[3 * n + i] = p.ux;
  q.pred[4 * n + i] = p.uy;
  q.pred[5 * n + i] = p.uz;
  q.xc[i] = (signed char)p.cross;
}

// Every instance's Lees-Edwards geometry at the time adv steps on, by one
// block (its fmod takes microseconds: a block of its own, beside the
// particles').
__device__ __forceinline__ void set_step_geo(const Geo& g, const InstGeo* __restrict__ ig, const DevStatus* st, int adv,
                                             StepGeo* __restrict__ sg) {
  for (int k = threadIdx.x; k < g.K; k += blockDim.x) {
    const InstGeo& I = ig[k];
    const double off = le_offset(g, I, dev_nstep(st) + adv);
    const int fsh = le_shift_cells(I, off);
    const double offr = off - fsh * I.cs[0];
    StepGeo q;
    q.off = off;
    q.fsh = fsh;
    q.offr_hi = (float)offr;
    q.offr_lo = (float)(offr - (double)q.offr_hi);
    sg[k] = q;
  }
}

// The state of the operation's scans, by the threads of the grid.
__device__ __forceinline__ void reset_scans(const SortOut& q) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < q.scan_words; t += gridDim.x * blockDim.x)
    q.scan_status[t] = 0ull;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < q.row_words; t += gridDim.x * blockDim.x) q.row_sums[t] = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) q.scan_ticket[0] = 0;
}
