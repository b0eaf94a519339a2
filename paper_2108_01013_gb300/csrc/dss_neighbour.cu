// Symmetric (half-stencil) fixed-radius near-neighbour enumeration
// (Sec. II A, Fig. 5): each pair is found exactly once, by its owner, and
// written into the owner's fixed-capacity row (capacity M, the shell
// estimate of Sec. II A), in a fixed visiting order.
//
// The decision uses an FP32 conservative prefilter on cell-local coordinates;
// candidates within the rounding band of the cutoff are decided by the exact
// FP64 predicate, so the pair set is the FP64 brute-force set bit for bit.
//
// Two searches give the same pairs, and write them into the owners' rows.  On
// sparse grids and with size classes a thread walks its owner's stencil
// (k_enumerate, k_enumerate_classes); on crowded grids a block takes the owners
// of a few cells and stages the candidates of their stencils in shared memory
// (k_enumerate_seg).  k_rows then scans the rows' lengths (the pair offsets of
// each owner) and writes the compact pair arrays.  With the scan at the end of
// the walk, by look-back over a tile per warp, thousands of tiles finished
// together and each walked back over all before it (a pass of its own: the batch
// of 64 333 -> 316 us a step).
#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "dss_internal.cuh"

namespace {
constexpr int kThreads = 128;
constexpr int kRows = 5;           // rows of cells in the half stencil, a warp each
constexpr int kTile = 128;         // candidates of a row staged at a time
constexpr int kSegMax = 28;        // cells of a segment (its stencil rows span three more)
constexpr int kRowThreads = 256;   // row pass
constexpr int kRowGroup = 16;      // tiles of a group

// Cutoffs of the pair (i, j) in FP32, linear in the radii: s = (a_i + a_j) sc + sd
// (the listing range) and (a_i + a_j) lc + ld (the lubrication range, row
// order only).  ECH: the listing range is the larger of s and a_i + a_j + de.
// The FP32 cutoff is within a few ulp of the exact one, far inside the margin.
struct EnumCut {
  float sc, sd, lc, ld, de;
};

// Per-owner state of the enumeration; everything the candidate loop reads is
// held in registers.
struct EnumCtx {
  const float4* __restrict__ posf;
  float4 pi;
  float sc, sa;     // cutoff of pair (i, j): s = a_j sc + sa (a_i + a_j + delta)
  float sa2;        // with electro-chemical forces the cutoff is max(s, a_j + sa2)
  float m2;         // r^2 margin of the FP32 decision
  float hx, hy, hz; // half box: a separation beyond it is decided exactly
  bool img;         // the stencil reaches past half the box along some axis
  int M;
  int cnt;
  int band;
  int* row;
  // exact FP64 decision
  const Geo* g;
  const InstGeo* I;
  const StateBuf* s;
  double off;
  int i;
};

__device__ __forceinline__ void enum_init(EnumCtx& e, const Geo& g, const InstGeo& I, const StateBuf& s,
                                          const float4* __restrict__ posf, int i, double off, int* row,
                                          int reach, const EnumCut& q) {
  e.posf = posf;
  e.pi = posf[i];
  e.sc = q.sc;
  e.sa = fmaf(e.pi.w, q.sc, q.sd);
  e.sa2 = e.pi.w + q.de;
  e.m2 = I.r2_margin;
  e.hx = I.halfLf[0];
  e.hy = I.halfLf[1];
  e.hz = I.halfLf[2];
  // a stencil cell is at most reach+1 cells away along y and z and, across
  // y = L_y, reach+2 along x: separations stay below half the box when the
  // box is wider than twice that (plus one cell of slack)
  e.img = I.nc[0] < 2 * reach + 5 || I.nc[1] < 2 * reach + 3 || I.nc[2] < 2 * reach + 3;
  e.M = g.M;
  e.cnt = 0;
  e.band = 0;
  e.row = row;
  e.g = &g;
  e.I = &I;
  e.s = &s;
  e.off = off;
  e.i = i;
}

// One candidate j of owner i (positions relative to the candidate cell's
// origin): FP32 decision on cell-local coordinates, certainly a pair,
// certainly not, or (within the margin of the cutoff, or past half the box)
// the exact FP64 predicate; a pair is appended to the row.
template <bool ECH>
__device__ __forceinline__ void take_candidate(EnumCtx& e, float4 pj, int j, float px, float py, float pz) {
  const float dx = pj.x - px, dy = pj.y - py, dz = pj.z - pz;
  float sv = fmaf(pj.w, e.sc, e.sa);
  if (ECH) sv = fmaxf(sv, pj.w + e.sa2);
  const float t = fmaf(-sv, sv, fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
  // nearly every candidate lies beyond the cutoff by more than the margin:
  // one test and out (the half-box image test only on boxes narrower than
  // the stencil)
  if (t > e.m2 && !e.img) return;
  int dec;
  if (e.img && (fabsf(dx) > e.hx || fabsf(dy) > e.hy || fabsf(dz) > e.hz))
    dec = -1;
  else
    dec = t < -e.m2 ? 1 : (t > e.m2 ? 0 : -1);
  if (dec < 0) {
    ++e.band;
    const StateBuf& s = *e.s;
    const int n = e.g->n, i = e.i;
    dec = exact_is_pair(*e.g, *e.I, e.off, s.x[i], s.x[n + i], s.x[2 * n + i], s.a[i], s.x[j],
                        s.x[n + j], s.x[2 * n + j], s.a[j]) ? 1 : 0;
  }
  if (dec) {
    if (e.cnt < e.M) e.row[e.cnt] = j;
    ++e.cnt;
  }
}

// Visits the candidates [jb, je) of one stencil cell (origin displaced by
// (cxo, cyo, czo) from the owner's cell) in order.
template <bool ECH>
__device__ __forceinline__ void scan_range(EnumCtx& e, int jb, int je, float cxo, float cyo, float czo) {
  const float px = e.pi.x - cxo, py = e.pi.y - cyo, pz = e.pi.z - czo;
  for (int j = jb; j < je; ++j) take_candidate<ECH>(e, __ldg(e.posf + j), j, px, py, pz);
}

// Sums of the rows' lengths, kept for the row pass: over its tiles of 2^shift
// owners, and over kRowGroup tiles each.
struct RowSums {
  int* tile;
  int* group;
  int shift;
};

__device__ __forceinline__ void add_rows(const RowSums& R, int t, int v) {
  atomicAdd(&R.tile[t], v);
  atomicAdd(&R.group[t / kRowGroup], v);
}

// The length of the owner's row, its warp's sum (a warp lies in one tile), and
// the exact decisions counted.
__device__ __forceinline__ void finish_row(const EnumCtx& e, int i, int n, int* __restrict__ count, const RowSums& R,
                                           DevStatus* st) {
  if (i < n) count[i] = e.cnt;
  const int sum = __reduce_add_sync(0xffffffffu, i < n ? min(e.cnt, e.M) : 0);
  if ((threadIdx.x & 31) == 0 && sum) add_rows(R, i >> R.shift, sum);
  const int b = __reduce_add_sync(0xffffffffu, i < n ? e.band : 0);
  if ((threadIdx.x & 31) == 0 && b) atomicAdd(&st->w[ST_BAND], b);
}

template <bool ECH>
__global__ void __launch_bounds__(kThreads, 8)
k_enumerate(Geo g, const InstGeo* __restrict__ ig, const StepGeo* __restrict__ sgk, StateBuf s,
            const float4* __restrict__ posf, const int* __restrict__ cellid,
            const int* __restrict__ cell_start, ListBuf L, RowSums R, DevStatus* st, EnumCut q) {
  dep_wait();
  if (dev_err(st)) return;
  const int i = blockIdx.x * kThreads + threadIdx.x;
  const int n = g.n;
  EnumCtx e;
  e.cnt = 0;
  e.band = 0;
  if (i < n) {
    const int inst = s.inst[i];
    const InstGeo& I = ig[inst];
    const StepGeo sg = sgk[inst];
    enum_init(e, g, I, s, posf, i, sg.off, L.list + (int64_t)i * g.Ms, 1, q);
    const int fsh = sg.fsh;
    const float offr = sg.offr_hi;
    const int nx = I.nc[0], ny = I.nc[1], nz = I.nc[2];
    const int cb = I.cell_base;
    const int c = cellid[i] - cb;
    const int cx = c % nx, cy = (c / nx) % ny, cz = c / (nx * ny);
    // neighbouring cell coordinates by conditional wraps (no integer
    // division in the stencil walk; every offset below stays within one box)
    const int xm = cx == 0 ? nx - 1 : cx - 1, xp = cx + 1 == nx ? 0 : cx + 1;
    const int zm = cz == 0 ? nz - 1 : cz - 1, zp = cz + 1 == nz ? 0 : cz + 1;
    // the bounds of a row's cells are read together, and before the row above
    // is scanned (one wait where every cell had its own: 100k 71.9 -> 70.9 us a
    // step)
    const bool le = cy == ny - 1;
    const int fshx = le ? 2 + fsh : 1;       // offset of the first cell of layer y+1
    const int yrow = (le ? 0 : cy + 1) * nx;
    const int xs = le ? wrapi(cx - fshx, nx) : xm;
    const int x1 = xs + 1 == nx ? 0 : xs + 1, x2 = x1 + 1 == nx ? 0 : x1 + 1, x3 = x2 + 1 == nx ? 0 : x2 + 1;
    const int* __restrict__ own = cell_start + cb + (cz * ny + cy) * nx;
    const int* __restrict__ r0 = cell_start + cb + (zp * ny + cy) * nx;
    const int own_end = own[cx + 1], nxt = own[xp], nxt_end = own[xp + 1];
    int lo0 = r0[xm], hi0 = r0[xm + 1], lo1 = r0[cx], hi1 = r0[cx + 1], lo2 = r0[xp], hi2 = r0[xp + 1], lo3 = 0, hi3 = 0;
    // own cell (partners after i) and the cell x+1
    scan_range<ECH>(e, i + 1, own_end, 0.f, 0.f, 0.f);
    scan_range<ECH>(e, nxt, nxt_end, I.csf[0], 0.f, 0.f);
    // layer y, z+1: three x cells; layer y+1: 3x3 cells, or across y = L_y the
    // 4 x cells covering the image range shifted by the Lees-Edwards offset
    float sx = -I.csf[0], sy = 0.f, sz = I.csf[2];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int a0 = lo0, b0 = hi0, a1 = lo1, b1 = hi1, a2 = lo2, b2 = hi2, a3 = lo3, b3 = hi3;
      if (r < 3) {
        const int qz = r == 0 ? zm : (r == 1 ? cz : zp);
        const int* __restrict__ p = cell_start + cb + qz * ny * nx + yrow;
        lo0 = p[xs]; hi0 = p[xs + 1]; lo1 = p[x1]; hi1 = p[x1 + 1]; lo2 = p[x2]; hi2 = p[x2 + 1];
        if (le) { lo3 = p[x3]; hi3 = p[x3 + 1]; }
      }
      scan_range<ECH>(e, a0, b0, sx, sy, sz);
      scan_range<ECH>(e, a1, b1, sx + I.csf[0], sy, sz);
      scan_range<ECH>(e, a2, b2, sx + 2.f * I.csf[0], sy, sz);
      if (r > 0 && le) scan_range<ECH>(e, a3, b3, sx + 3.f * I.csf[0], sy, sz);
      if (r == 0) {
        sx = le ? fmaf(-2.f, I.csf[0], offr) : -I.csf[0];
        sy = I.csf[1];
        sz = -I.csf[2];
      } else {
        sz += I.csf[2];
      }
    }
  }
  finish_row(e, i, n, L.count, R, st);
}

// Size classes (Sec. II A: cells smaller than 2 a_max, a larger stencil for
// the larger particles).  Owner i of class c takes the partners of its own
// class from the half stencil of reach R = rtab[c][c] (own bin after i; the
// rest of the own row in +x; the rows z+1..z+R of its y layer; the layers
// y+1..y+R), and the partners of every smaller class c2 from the full stencil
// of reach rtab[c][c2] in that class's layer of bins: each pair is found
// once, by its larger member (or by the half stencil within a class).  Rows
// crossing y = L_y (either way) cover the x range shifted by the
// Lees-Edwards offset.
template <bool ECH>
__global__ void __launch_bounds__(kThreads, 8)
k_enumerate_classes(Geo g, const InstGeo* __restrict__ ig, const StepGeo* __restrict__ sgk, StateBuf s,
                    const float4* __restrict__ posf, const int* __restrict__ cellid,
                    const int* __restrict__ cell_start, ListBuf L, RowSums R, DevStatus* st, EnumCut q) {
  dep_wait();
  if (dev_err(st)) return;
  const int i = blockIdx.x * kThreads + threadIdx.x;
  const int n = g.n;
  EnumCtx e;
  e.cnt = 0;
  e.band = 0;
  if (i < n) {
    const int inst = s.inst[i];
    const InstGeo& I = ig[inst];
    const StepGeo sg = sgk[inst];
    enum_init(e, g, I, s, posf, i, sg.off, L.list + (int64_t)i * g.Ms, g.reach, q);
    const int fsh = sg.fsh;
    const float offr = sg.offr_hi;
    const int nx = I.nc[0], ny = I.nc[1], nz = I.nc[2];
    const int layer = I.ncell_layer;
    const int cls = s.cls[i];
    const int c = (cellid[i] - I.cell_base) % layer;
    const int cx = c % nx, cy = (c / nx) % ny, cz = c / (nx * ny);
    // own bin, partners after i
    scan_range<ECH>(e, i + 1, cell_start[cellid[i] + 1], 0.f, 0.f, 0.f);
    for (int c2 = cls; c2 >= 0; --c2) {
      const int R = g.rtab[cls][c2];
      const bool half = c2 == cls;
      const int lb = I.cell_base + c2 * layer;
      for (int oy = half ? 0 : -R; oy <= R; ++oy) {
        const int yy = cy + oy;
        const int le = yy >= ny ? 1 : (yy < 0 ? -1 : 0);
        const int qy = le == 1 ? yy - ny : (le == -1 ? yy + ny : yy);
        for (int oz = (half && oy == 0) ? 0 : -R; oz <= R; ++oz) {
          const int qz = wrapi(cz + oz, nz);
          int xa, xb;
          if (half && oy == 0 && oz == 0) {
            xa = 1;
            xb = R;
          } else if (le == 1) {
            xa = -R - 1 - fsh;
            xb = R - fsh;
          } else if (le == -1) {
            xa = -R + fsh;
            xb = R + 1 + fsh;
          } else {
            xa = -R;
            xb = R;
          }
          // the row's cells are adjacent bins (split where x wraps): one
          // candidate range per piece, most of them empty on small cells
          const int rowq = lb + (qz * ny + qy) * nx;
          int ox = xa;
          while (ox <= xb) {
            const int x0 = wrapi(cx + ox, nx);
            const int m = min(xb - ox + 1, nx - x0);
            const int q0 = rowq + x0;
            const int lo = cell_start[q0], hi = cell_start[q0 + m];
            if (lo < hi) {
              int k = 0, kend = cell_start[q0 + 1];
              float cxo, cyo, czo;
              stencil_shift(I, ox, oy, oz, le, fsh, offr, cxo, cyo, czo);
              for (int j = lo; j < hi; ++j) {
                if (j >= kend) {
                  do {
                    ++k;
                    kend = cell_start[q0 + k + 1];
                  } while (j >= kend);
                  stencil_shift(I, ox + k, oy, oz, le, fsh, offr, cxo, cyo, czo);
                }
                scan_range<ECH>(e, j, j + 1, cxo, cyo, czo);
              }
            }
            ox += m;
          }
        }
      }
    }
  }
  finish_row(e, i, n, L.count, R, st);
}

// Two FP32 values in one register pair, for the packed instructions.
__device__ __forceinline__ uint64_t pk2(float a, float b) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
__device__ __forceinline__ float2 upk2(uint64_t v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// A separation beyond half the box is not the nearest image's; that one, the
// box less it, can be a pair's only below a cell's edge, which no cutoff
// exceeds: separations beyond the box less one cell (and a thousandth for the
// rounding) are decided exactly.
__device__ __forceinline__ float exact_beyond(const InstGeo& I, int d) {
  return fmaxf(I.halfLf[d], 2.f * I.halfLf[d] - 1.001f * I.csf[d]);
}

// Candidate k of a row staged two by two: {x, x', y, y'}, {z, z', a, a'}.
__device__ __forceinline__ float4 staged(const float4* row, int k) {
  const float* f = reinterpret_cast<const float*>(row) + 8 * (k >> 1) + (k & 1);
  return make_float4(f[0], f[2], f[4], f[6]);
}

// Exact decision of (i, j) (out of line: about one candidate in a thousand).
__device__ __noinline__ bool decide_exact(const Geo& g, const InstGeo& I, const StateBuf& s, double off, int i,
                                          int j) {
  const int n = g.n;
  return exact_is_pair(g, I, off, s.x[i], s.x[n + i], s.x[2 * n + i], s.a[i], s.x[j], s.x[n + j], s.x[2 * n + j],
                       s.a[j]);
}

// ------------------------------------------------------------------------
// Segment walk.  One block per segment: seg consecutive x cells of one row of
// cells, as many as hold about 26 particles (one cell on dense grids, then
// shared by several blocks), a lane per owner.  The half stencil of the
// segment is five rows of adjacent cells, each one or (across x = L_x) two
// pieces of the sorted order: its own row from the segment on, the z+1 row and
// the three rows of layer y+1 (across y = L_y one x cell more, shifted by the
// Lees-Edwards offset).  A warp takes one of them: it reads the cell offsets,
// stages the particles in shared memory relative to the segment's origin,
// kTile at a time, and each lane runs over its own cells' part of them.
//
// Two candidates are staged and screened together (packed FP32 arithmetic, the
// same roundings): 7 instructions a candidate instead of 11
// (1M 197 -> 187 us, Table 5 178 -> 174).
//
// What bounds it is the issue slots (2.4 to 2.9 instructions a cycle and SM):
// a candidate is loaded once for 32 owners instead of once for each, and costs
// a lane 7 instructions, one of them a shared load; the set-up of a block is
// worth half a pass of 32 owners.  Against the walk by owner with the same
// screen (one box, mixed precision, with the row pass): Table 5 with the 4 a0
// range (128 per cell, 2.9M pairs) 312 -> 167 us, 1M log-uniform [1, 10] (7.1
// per cell) 220 -> 178, the 100k packing with the 1 a0 range (4.1 per cell) 40
// -> 34.  On sparse grids the set-up does not pay: 100k (1.7 per cell) 28
// against 37 us, a batch of 64 (1.8) 106 against 202.
//
// The decision: u = r^2 - s^2 in FP32, its sign bit shifted into a mask, 32
// candidates at a time without a branch, with the smallest |u| beside it.  A
// lane whose smallest |u| lies within the margin (1e-4 cell^2; positions up
// to 31 cells from the origin round to 2e-6 cell, u near the cutoff to
// 1e-5 cell^2) takes those candidates again with the exact FP64 predicate.  A
// box as narrow as the stencil (NARROW) takes every candidate of such a row
// again, and those that may be nearer by another image exactly too.  (With every
// separation beyond half the box decided exactly, and every candidate taken
// again in boxes of up to six cells, 12,000 spheres of Table 5 in 4^3 cells took
// 594 us a step instead of 208, 30,000 in 6^3 257 instead of 223.)
//
// An owner's row lists the pairs of the five rows of cells in turn, ascending
// within each (tile by tile on dense grids): the warps exchange the owners'
// counts and write their own part.  SPLIT (pairs listed beyond the lubrication
// range, with electro-chemical forces): pairs within the lubrication range by
// an FP32 test go to the row's front, the others to its back from the end;
// k_rows closes the row up.
// ------------------------------------------------------------------------
// What a block of the staged search keeps in shared memory.
struct SegShared {
  float4 c[kRows][kTile + 4];
  int j[kRows][kTile];
  int off[kRows][32];
  int len[kRows];
  int cnt[2][kRows][32];      // pairs of each owner in each row (near ones << 16: SPLIT)
  int4 par[kRows];            // rows: bin of their x = 0, x of their first cell, cells, image across y
  int seg[4];                 // first bin, cells, part, first owner
  int far;                    // ST_LONG, then the group to take after the block's own owners (-1: none is left)
};

// The segment from x0 on in a row of cells: its half stencil's rows, a lane each
// (by one warp).
__device__ __forceinline__ void set_segment(SegShared& sh, const InstGeo& I, int fsh, int row, int x0, int part) {
  const int nx = I.nc[0], ny = I.nc[1], nz = I.nc[2], lane = threadIdx.x & 31;
  const int cz = row / ny, cy = row - cz * ny;
  const int bxe = min(I.enum_seg, nx - x0);
  const bool img = lane >= 2 && cy == ny - 1;
  int xf = lane == 0 ? x0 : (img ? wrapi(x0 - 2 - fsh, nx) : x0 - 1);
  if (xf < 0) xf += nx;
  const int qy = lane < 2 ? cy : (cy == ny - 1 ? 0 : cy + 1);
  int qz = lane == 0 ? cz : (lane == 1 ? cz + 1 : cz + lane - 3);
  qz = qz < 0 ? nz - 1 : (qz == nz ? 0 : qz);
  if (lane < kRows)
    sh.par[lane] = make_int4(I.cell_base + (qz * ny + qy) * nx, xf, bxe + (lane == 0 ? 1 : (img ? 3 : 2)), img);
  if (lane == 0) {
    sh.seg[0] = I.cell_base + row * nx + x0;
    sh.seg[1] = bxe;
    sh.seg[2] = part;
  }
}

// Owners of a segment of len that its own blocks take (and on to a multiple of
// 32 in the sorted order): all, up to seven passes more than its average blocks
// have; of a longer one, whose stencil rows are long too, those blocks' alone.
__host__ __device__ __forceinline__ int seg_long(const InstGeo& I) { return 32 * I.enum_subs + 224; }
__device__ __forceinline__ int seg_limit(const InstGeo& I, int len) {
  return len <= seg_long(I) ? len : 32 * I.enum_subs;
}

// Group k of those a block looks at for owners beyond their segment's limit: 32 owners
// from a multiple of 32 in the sorted order on, one in gridDim.x.
__device__ __forceinline__ int64_t far_group(int k) { return blockIdx.x + (int64_t)k * gridDim.x; }

// The segment in sh.par and sh.seg (complete at a barrier before the call): the
// owners of the block's part of it, or (grp >= 0) a group of its owners.
template <bool ECH, bool SPLIT, bool NARROW>
__device__ __forceinline__ void search_segment(
    SegShared& sh, const Geo& g, const InstGeo& I, const StepGeo& sg, const StateBuf& s,
    const float4* __restrict__ posf, const int* __restrict__ cellid, const int* __restrict__ cell_start,
    int* __restrict__ list, int* __restrict__ count, int* __restrict__ nnear, const RowSums& R, DevStatus* st,
    const EnumCut& q, int lane, int r, int grp) {
  const int nx = I.nc[0], ny = I.nc[1], nz = I.nc[2];
  // the warp's row: w cells from x = xf on, of the row of cells at rc
  const int4 par = sh.par[r];
  const int rc = par.x, xf = par.y, w = par.z;
  const bool le = par.w != 0;
  // lane k: the boundary before its cell k, as a place in the row's sequence;
  // place p is particle first + p, or beyond x = L_x (p >= n1) first + wrap + p
  const int xk = xf + min(lane, w);
  int b = cell_start[rc + (xk <= nx ? xk : xk - nx)];
  const int first = __shfl_sync(0xffffffffu, b, 0);
  int n1 = INT_MAX, wrap = 0;
  if (xf + w > nx) {
    const int row0 = cell_start[rc];
    n1 = cell_start[rc + nx] - first;
    wrap = row0 - n1 - first;
    b = xk <= nx ? b - first : b - row0 + n1;
  } else {
    b -= first;
  }
  sh.off[r][lane] = b;
  const int len = __shfl_sync(0xffffffffu, b, w);
  if (lane == 0) {
    sh.len[r] = len;
    if (r == 0) sh.seg[3] = first;
  }
  __syncthreads();
  const int c0 = sh.seg[0], part = sh.seg[2], hs = sh.seg[3], he = hs + sh.off[0][sh.seg[1]];
  const int o_beg = grp >= 0 ? 32 * grp : hs + 32 * (part < 0 ? -1 - part : part);
  const int o_end = min(grp >= 0 || part >= 0 ? o_beg + 32 : (hs + seg_limit(I, he - hs) + 31) & ~31, he);
  const int most = max(max(max(sh.len[0], sh.len[1]), max(sh.len[2], sh.len[3])), sh.len[4]);
  const float kx0 = r == 0 ? 0.f : (le ? -2.f : -1.f), sx = le ? sg.offr_hi : 0.f;
  const float sy = r < 2 ? 0.f : I.csf[1];
  const float sz = r == 0 ? 0.f : (r == 1 ? I.csf[2] : (float)(r - 3) * I.csf[2]);
  // rows of cells that reach past exact_beyond (two cells, along x three across
  // y = L_y)
  const bool img = NARROW && (nx < (le ? 5 : 4) || ny < 4 || nz < 4);
  const float m2 = I.r2_margin;
  int buf = 0, band = 0;
  for (int o0 = o_beg; o0 < o_end; o0 += 32) {
    // the lane's owner and its part [lo, hi) of the row
    const int i = o0 + lane;
    const bool in = i < o_end;
    float px = 0.f, py = 0.f, pz = 0.f, pa = 0.f, sa = 0.f;
    int lo = 0, hi = 0;
    if (in) {
      const float4 p = posf[i];
      const int kx = cellid[i] - c0;
      px = fmaf((float)kx, I.csf[0], p.x);
      py = p.y;
      pz = p.z;
      pa = p.w;
      sa = fmaf(p.w, q.sc, q.sd);
      lo = r == 0 ? i - hs + 1 : sh.off[r][kx];
      hi = sh.off[r][kx + (r == 0 ? 2 : (le ? 4 : 3))];
    }
    const uint64_t npx = pk2(-px, -px), npy = pk2(-py, -py), npz = pk2(-pz, -pz);
    const uint64_t sc2 = pk2(q.sc, q.sc), sa2 = pk2(sa, sa), nsc2 = pk2(-q.sc, -q.sc), nsa2 = pk2(-sa, -sa);
    const uint64_t se2 = pk2(pa + q.de, pa + q.de);
    int* rw = list + (int64_t)i * g.Ms;
    int pairs = 0, near = 0;    // of the owner, in the tiles so far
    for (int t0 = 0; t0 < most; t0 += kTile) {
      const int t1 = min(t0 + kTile, len);
      if (o0 == o_beg || most > kTile) {     // (a single tile stays for the next owners)
        __syncwarp();
        for (int p0 = t0; p0 < t1; p0 += 32) {
          const int p = p0 + lane;
          float4 c = make_float4(1e15f, 1e15f, 1e15f, 0.f);   // beside an odd last one
          if (p < t1) {
            const int j = first + p + (p < n1 ? 0 : wrap);
            c = __ldg(posf + j);
            int kc = __ldg(cellid + j) - rc - xf;
            if (kc < 0) kc += nx;
            c.x += fmaf((float)kc + kx0, I.csf[0], sx);
            c.y += sy;
            c.z += sz;
            sh.j[r][p - t0] = j;
          }
          // even lanes hold the two particles' x and y, odd ones z and a
          const float va = __shfl_xor_sync(0xffffffffu, lane & 1 ? c.x : c.z, 1);
          const float vb = __shfl_xor_sync(0xffffffffu, lane & 1 ? c.y : c.w, 1);
          if ((p & ~1) < t1)
            sh.c[r][p - t0] = lane & 1 ? make_float4(va, c.z, vb, c.w) : make_float4(c.x, va, c.y, vb);
        }
        __syncwarp();
      }
      // the lane's part of the tile, from an even place on
      const int a0 = max(lo, t0) - t0, z = min(hi, t1) - t0, a = a0 & ~1;
      const int words = __reduce_max_sync(0xffffffffu, (z - a + 31) >> 5);
      unsigned hit[kTile / 32];
#pragma unroll
      for (int h = 0; h < kTile / 32; ++h) {
        hit[h] = 0u;
        if (h >= words) continue;
        const int m = min(32, z - a - 32 * h);
        if (m <= 0) continue;
        const float4* __restrict__ c = &sh.c[r][a + 32 * h];
        float least = __int_as_float(0x7f800000);
        int n = 0;
        do {
#pragma unroll
          for (int u = 0; u < 4; u += 2) {
            const float4 xy = c[n + u], za = c[n + u + 1];   // up to three past the end: masked off below
            const uint64_t dx = add2(pk2(xy.x, xy.y), npx), dy = add2(pk2(xy.z, xy.w), npy);
            const uint64_t dz = add2(pk2(za.x, za.y), npz), aj = pk2(za.z, za.w);
            const uint64_t r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
            const uint64_t sv = fma2(aj, sc2, sa2);
            float2 t;
            if (ECH) {
              const float2 s1 = upk2(sv), s2 = upk2(add2(aj, se2)), rr = upk2(r2);
              const float m0 = fmaxf(s1.x, s2.x), m1 = fmaxf(s1.y, s2.y);
              t = make_float2(fmaf(-m0, m0, rr.x), fmaf(-m1, m1, rr.y));
            } else {
              t = upk2(fma2(fma2(aj, nsc2, nsa2), sv, r2));
            }
            hit[h] = __funnelshift_l(__float_as_uint(t.x), hit[h], 1);
            hit[h] = __funnelshift_l(__float_as_uint(t.y), hit[h], 1);
            least = fminf(least, fminf(fabsf(t.x), fabsf(t.y)));
          }
          n += 4;
        } while (n < m);
        hit[h] <<= 32 - n;                          // candidate b at bit 31 - b
        unsigned all = ~(m < 32 ? 0xffffffffu >> m : 0u);
        if (h == 0 && a != a0) all &= 0x7fffffffu;
        hit[h] &= all;
        if (least <= m2 || img) {
          for (unsigned left = all; left;) {
            const int e = __clz(left);
            const unsigned bit = 0x80000000u >> e;
            left &= ~bit;
            const float4 pj = staged(c, e);
            const float dx = pj.x - px, dy = pj.y - py, dz = pj.z - pz;
            float sv = fmaf(pj.w, q.sc, sa);
            if (ECH) sv = fmaxf(sv, pj.w + (pa + q.de));
            const float t = fmaf(-sv, sv, fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
            if (!(fabsf(t) > m2) ||
                (img && (fabsf(dx) > exact_beyond(I, 0) || fabsf(dy) > exact_beyond(I, 1) || fabsf(dz) > exact_beyond(I, 2)))) {
              ++band;
              if (decide_exact(g, I, s, sg.off, i, sh.j[r][a + 32 * h + e])) hit[h] |= bit;
              else hit[h] &= ~bit;
            }
          }
        }
      }
      int mine = 0;
      unsigned nrm[kTile / 32];
#pragma unroll
      for (int h = 0; h < kTile / 32; ++h) {
        nrm[h] = 0u;
        if (h >= words) continue;
        mine += __popc(hit[h]);
        if (SPLIT) {
          for (unsigned left = hit[h]; left;) {
            const int e = __clz(left);
            left &= ~(0x80000000u >> e);
            const float4 pj = staged(sh.c[r], a + 32 * h + e);
            const float dx = pj.x - px, dy = pj.y - py, dz = pj.z - pz;
            const float sl = fmaf(pa + pj.w, q.lc, q.ld);
            if (fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < sl * sl) nrm[h] |= 0x80000000u >> e;
          }
          mine += __popc(nrm[h]) << 16;
        }
      }
      sh.cnt[buf][r][lane] = mine;
      __syncthreads();
      int at = 0, tot = 0;
#pragma unroll
      for (int v = 0; v < kRows; ++v) {
        if (v == r) at = tot;
        tot += sh.cnt[buf][v][lane];
      }
      buf ^= 1;
      // the warp's part of the owner's row
      int kn = SPLIT ? near + (at >> 16) : pairs + at, kf = SPLIT ? pairs - near + (at & 0xffff) - (at >> 16) : 0;
#pragma unroll
      for (int h = 0; h < kTile / 32; ++h) {
        if (h >= words) break;
        for (unsigned left = hit[h]; left;) {
          const int e = __clz(left);
          const unsigned bit = 0x80000000u >> e;
          left &= ~bit;
          const int j = sh.j[r][a + 32 * h + e];
          if (SPLIT) {
            if (kn + kf < g.M) rw[nrm[h] & bit ? kn : g.M - 1 - kf] = j;
            if (nrm[h] & bit) ++kn; else ++kf;
          } else {
            if (kn < g.M) rw[kn] = j;
            ++kn;
          }
        }
      }
      pairs += SPLIT ? tot & 0xffff : tot;
      near += SPLIT ? tot >> 16 : 0;
    }
    if (r == 0) {
      if (in) {
        count[i] = pairs;
        if (SPLIT) nnear[i] = near;
      }
      // (owners from o0 on: in one tile or two)
      const int t = o0 >> R.shift, v = in ? min(pairs, g.M) : 0;
      const int s0 = __reduce_add_sync(0xffffffffu, i >> R.shift == t ? v : 0);
      const int s1 = __reduce_add_sync(0xffffffffu, i >> R.shift == t ? 0 : v);
      if (lane == 0 && s0) add_rows(R, t, s0);
      if (lane == 0 && s1) add_rows(R, t + 1, s1);
    }
  }
  if (__any_sync(0xffffffffu, band != 0)) {
    band = __reduce_add_sync(0xffffffffu, band);
    if (lane == 0) atomicAdd(&st->w[ST_BAND], band);
  }
}

// The owners beyond their segments' limits (few cells that hold most of the
// particles: segregated sizes), a group after another, after the block's own.
// Out of line and behind the sort's word that there are any (ST_LONG): looking
// for them in every block cost 2% of the search of 1M.  The search of 20,000
// small spheres beside a few large ones, a thousand to a cell of 512, 0.56 ms
// instead of 4.0 with such a cell's owners left to its last block (walked by
// owner 0.60); of 200,000 in 1000 cells 1.8 instead of 5.4 (4.4).
template <bool ECH, bool SPLIT, bool ONE, bool NARROW>
__device__ __noinline__ void search_far(
    SegShared& sh, const Geo& g, const InstGeo& I1, const InstGeo* __restrict__ ig, const StepGeo* __restrict__ sgk,
    const StateBuf& s, const float4* __restrict__ posf, const int* __restrict__ cellid,
    const int* __restrict__ cell_start, int* __restrict__ list, int* __restrict__ count, int* __restrict__ nnear,
    const RowSums& R, DevStatus* st, const EnumCut& q) {
  const int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
  for (int k = 0;; ++k) {
    __syncthreads();
    if (r == 0) {
      int found = -1;
      for (; found < 0 && 32 * far_group(k) < g.n; ++k) {
        const int64_t gk = far_group(k);
        const int i = 32 * (int)gk, inst = ONE ? 0 : s.inst[i];
        const InstGeo& I = ONE ? I1 : ig[inst];
        const int c = cellid[i], x = (c - I.cell_base) % I.nc[0], dx = x % I.enum_seg;
        const int hs = cell_start[c - dx], he = cell_start[c - dx + min(I.enum_seg, I.nc[0] - x + dx)];
        if (i - hs < seg_limit(I, he - hs)) continue;
        found = (int)gk;
        set_segment(sh, I, sgk[inst].fsh, (c - I.cell_base) / I.nc[0], x - dx, -1);
        break;
      }
      if (lane == 0) sh.far = found;
    }
    __syncthreads();
    const int grp = sh.far;
    if (grp < 0) return;
    const int inst = ONE ? 0 : s.inst[32 * grp];
    search_segment<ECH, SPLIT, NARROW>(sh, g, ONE ? I1 : ig[inst], sgk[inst], s, posf, cellid, cell_start, list, count,
                                       nnear, R, st, q, lane, r, grp);
  }
}

template <bool ECH, bool SPLIT, bool ONE, bool NARROW>
__global__ void __launch_bounds__(32 * kRows, 7)
k_enumerate_seg(const __grid_constant__ Geo g, const __grid_constant__ InstGeo I1, const InstGeo* __restrict__ ig,
            const StepGeo* __restrict__ sgk, const __grid_constant__ StateBuf s, const float4* __restrict__ posf,
            const int* __restrict__ cellid, const int* __restrict__ cell_start, int* __restrict__ list,
            int* __restrict__ count, int* __restrict__ nnear, const int* __restrict__ blk_inst,
            const __grid_constant__ RowSums R, DevStatus* st, const __grid_constant__ EnumCut q) {
  dep_wait();
  __shared__ SegShared sh;
  if (dev_err(st)) return;
  int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
  asm volatile("" : "+r"(lane), "+r"(r));     // kept, not taken anew in every loop
  const int inst = ONE ? 0 : blk_inst[blockIdx.x];
  const InstGeo& I = ONE ? I1 : ig[inst];
  const StepGeo sg = sgk[inst];
  if (threadIdx.x == 32) sh.far = st->w[ST_LONG];
  if (r == 0) {
    // the first warp finds the segment
    unsigned item = blockIdx.x - (ONE ? 0 : I.enum_blk);
    const int subs = I.enum_subs;
    int sub = 0;
    if (subs > 1) {
      const unsigned h = item / (unsigned)subs;
      sub = (int)(item - h * subs);
      item = h;
    }
    const int row = (int)(item / (unsigned)I.enum_hx);
    set_segment(sh, I, sg.fsh, row, ((int)item - row * I.enum_hx) * I.enum_seg, sub + 1 < subs ? sub : -1 - sub);
  }
  __syncthreads();
  search_segment<ECH, SPLIT, NARROW>(sh, g, I, sg, s, posf, cellid, cell_start, list, count, nnear, R, st, q, lane, r,
                                     -1);
  if (sh.far)
    search_far<ECH, SPLIT, ONE, NARROW>(sh, g, I1, ig, sgk, s, posf, cellid, cell_start, list, count, nnear, R, st, q);
}

// Row pass: counters, the id <-> row maps, the exclusive scan of the row
// lengths and the compact pair arrays (owner and partner of every pair in owner
// order, the order the pair kernel deals them out in), written by the block
// together, coalesced.  A tile's first pair is the sum of the groups and tiles
// before it, which the search left: no block waits for another (with a
// look-back over the tiles a step of 20,000 spheres took 38.5 us instead of
// 36.2, Table 5's 446 instead of 440).  SPLIT rows are closed up in place here:
// the far block [M - far, M) moves down behind the near one, ascending, every
// entry read before any write reaches it (a source lies beyond its destination
// by the gap).  A kernel of its own:
// a row's place needs all rows before it.
// TILE: 256 owners, or 64 where rows are long (a block's pairs are what its
// time goes with).
template <bool SPLIT, int TILE>
__global__ void __launch_bounds__(kRowThreads)
k_rows(int n, int M, int Ms, int64_t pcap, const int* __restrict__ ids, const __grid_constant__ ListBuf L,
       const int* __restrict__ nnear, int* __restrict__ bw_count, const int* __restrict__ cellid,
       int* __restrict__ cell_more, RowSums R, DevStatus* st) {
  dep_wait();
  constexpr int kAhead = 4;                  // pairs a thread has in flight
  __shared__ int s_warp[kRowThreads / 32], s_pre[kRowThreads / 32];
  __shared__ int s_ex[TILE + 1], s_near[SPLIT ? TILE : 1];
  const int err = dev_err(st);
  const int tile = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int i0 = tile * TILE, i = i0 + threadIdx.x;
  const bool own = threadIdx.x < TILE && i < n;
  const int cnt = own ? L.count[i] : 0;
  const int v = min(cnt, M);
  if (SPLIT && own) s_near[threadIdx.x] = min(nnear[i], v);
  int pre = 0;
  for (int t = threadIdx.x; t < tile / kRowGroup; t += kRowThreads) pre += R.group[t];
  if (threadIdx.x < tile % kRowGroup) pre += R.tile[tile - 1 - threadIdx.x];
  pre = __reduce_add_sync(0xffffffffu, pre);
  int incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) {
    s_warp[wid] = incl;
    s_pre[wid] = pre;
  }
  if (__syncthreads_or(err)) return;
  int before = 0, total = 0, base = 0;
#pragma unroll
  for (int w = 0; w < kRowThreads / 32; ++w) {
    if (w < wid) before += s_warp[w];
    total += s_warp[w];
    base += s_pre[w];
  }
  if (threadIdx.x < TILE) s_ex[threadIdx.x] = before + incl - v;
  if (threadIdx.x == 0) {
    s_ex[TILE] = total;
    if (i0 + TILE >= n) L.start[n] = base + total;
  }
  __syncthreads();
  // pair t of the tile: its owner (the last whose row starts at or before t)
  // and its place there
  auto find = [&](int t, int& o, int& k, int& src) {
    o = 0;
#pragma unroll
    for (int step = TILE / 2; step >= 1; step >>= 1)
      if (s_ex[o + step] <= t) o += step;
    k = t - s_ex[o];
    src = k;
    if (SPLIT && k >= s_near[o]) src = M - (s_ex[o + 1] - s_ex[o]) + k;
  };
  int aj[kAhead], ao[kAhead], ak[kAhead];
#pragma unroll
  for (int r = 0; r < kAhead; ++r) {
    const int t = threadIdx.x + r * kRowThreads;
    aj[r] = -1;
    ao[r] = 0;
    ak[r] = -1;
    if (t < total) {
      int k, src;
      find(t, ao[r], k, src);
      aj[r] = L.list[(int64_t)(i0 + ao[r]) * Ms + src];
      if (src != k) ak[r] = k;
    }
  }
  const int wmax = __reduce_max_sync(0xffffffffu, cnt);
  if (lane == 0 && wmax > *(volatile int*)&st->w[ST_MAXROW]) atomicMax(&st->w[ST_MAXROW], wmax);
  if (own) {
    if (cnt > M) {
      L.count[i] = M;
      set_err(st, DSS_ERR_CAPACITY);
    }
    bw_count[i] = 0;
    const int id = ids[i];
    L.slot_of_id[id] = i;
    L.id_of_slot[i] = id;
    L.start[i] = base + before + incl - v;
  }
  if (SPLIT) __syncthreads();
#pragma unroll
  for (int r = 0; r < kAhead; ++r) {
    const int t = threadIdx.x + r * kRowThreads;
    if (t < total) {
      if (base + t < pcap) {
        L.pj[base + t] = aj[r];
        L.pown[base + t] = i0 + ao[r];
      }
      if (SPLIT && ak[r] >= 0) L.list[(int64_t)(i0 + ao[r]) * Ms + ak[r]] = aj[r];
    }
  }
  if (own && st->w[ST_CELL]) cell_more[cellid[i]] = 0;   // the sort's chains, for the next one
  for (int t0 = kAhead * kRowThreads; t0 < total; t0 += kRowThreads) {
    const int t = t0 + threadIdx.x;
    int o = 0, k = 0, src = 0, j = 0;
    if (t < total) {
      find(t, o, k, src);
      j = L.list[(int64_t)(i0 + o) * Ms + src];
    }
    if (SPLIT) __syncthreads();
    if (t < total) {
      if (base + t < pcap) {
        L.pj[base + t] = j;
        L.pown[base + t] = i0 + o;
      }
      if (SPLIT && src != k) L.list[(int64_t)(i0 + o) * Ms + k] = j;
    }
  }
}
}  // namespace

// Tiles of 64 owners (the smaller ones), and with their groups.
void row_sum_words(int n, int& tiles, int& words) {
  tiles = (n + 63) / 64;
  words = tiles + (tiles + kRowGroup - 1) / kRowGroup;
}

// Expected passes of 32 owners over a segment of mean owners (Poisson counts).
static double seg_passes(double mean) {
  double e = 0.0, p = std::exp(-mean);   // p: probability of exactly k owners
  for (int k = 1; k <= 4 * (int)mean + 64; ++k) {
    p *= mean / k;
    e += p * ((k + 31) / 32);
  }
  return e;
}

// The enumeration's kernel and launch for the current grid.  Grids of fewer
// than four particles a cell, and of size classes, are walked by owner (the
// two searches meet between 1.8 and 4.1 per cell, see k_enumerate_seg), except
// single systems of up to 360 owners per SM: there the walk's chain of loads
// is all that counts and five warps per segment shorten it (1,000 owners 19
// -> 13 us, 20,000 22 -> 16; a step of 40,000 45.7 -> 43.0, of 50,000 50.2 ->
// 48.4, of 65,000 57.9 -> 58.0, of 100,000 71.7 -> 76.1).
// Segments are cut so that the cost per owner is smallest: a block's set-up is
// worth about half a pass of 32 owners.  Cells of more than 26 particles are
// shared by as many blocks as hold their average and a quarter more.  Per
// instance: the segment's cells, the segments of a row of cells, the blocks of
// a segment, the first block.  Returns the number of blocks (and their
// instances, when asked for).
int64_t enum_plan(dss_handle* h, std::vector<int>* blk_inst) {
  const bool sparse = h->n < 4 * (int64_t)h->g.ncell && (h->K > 1 || h->n > 360 * (int64_t)h->sms);
  const bool empty = h->n * 4 < (int64_t)h->g.ncell;   // most segments would hold nobody
  h->enum_walk = h->g.nclass > 1 || h->tune_enum_unr == 1 || (h->tune_enum_unr == 0 && (sparse || empty));
  int64_t blk = 0;
  h->enum_narrow = false;
  h->enum_most_seg = 0;
  h->enum_long_seg = INT_MAX;
  if (blk_inst) blk_inst->clear();
  for (int k = 0; k < h->K; ++k) {
    InstGeo& I = h->ig_host[k];
    const double per = (double)h->inst_n[k] / (double)I.ncell;
    const int nx = I.nc[0];
    int hx = nx;
    h->enum_narrow |= nx < 5 || I.nc[1] < 4 || I.nc[2] < 4;
    I.enum_subs = 1;
    if (per > 26.0) {
      I.enum_subs = (int)std::min(std::ceil(1.25 * per / 32.0), 1024.0);
    } else {
      // (a row of the stencil holds each cell once: seg + 3 cells across
      // y = L_y; and a row of it fits one tile)
      double best = INFINITY;
      for (int seg = 1; seg <= std::min(kSegMax, nx - 3) && (seg == 1 || per * (seg + 2) < 0.9 * kTile); ++seg) {
        const int q = (nx + seg - 1) / seg;
        const double mean = per * nx / q, cost = (0.5 + seg_passes(mean)) / mean;
        if (cost < best) {
          best = cost;
          hx = q;
        }
      }
    }
    I.enum_hx = hx;
    I.enum_seg = (nx + hx - 1) / hx;
    h->enum_most_seg = std::max(h->enum_most_seg, I.enum_seg);
    h->enum_long_seg = std::min(h->enum_long_seg, seg_long(I));
    I.enum_blk = (int)blk;
    const int64_t items = (int64_t)hx * I.nc[1] * I.nc[2] * I.enum_subs;
    if (blk_inst && !h->enum_walk) blk_inst->insert(blk_inst->end(), (size_t)items, k);
    blk += items;
  }
  if (h->enum_walk) {
    blk = (h->n + kThreads - 1) / kThreads;
    h->enum_long_seg = INT_MAX;
  }
  h->enum_blocks = blk;
  return blk;
}

namespace {
// The staged search of one configuration (NARROW: some box is less than five
// cells wide along x or four along y or z; the others carry none of its code).
template <bool NARROW>
auto seg_kernel(bool ech, bool split, bool one) {
  return ech ? (split ? (one ? k_enumerate_seg<true, true, true, NARROW> : k_enumerate_seg<true, true, false, NARROW>)
                      : (one ? k_enumerate_seg<true, false, true, NARROW> : k_enumerate_seg<true, false, false, NARROW>))
             : (split ? (one ? k_enumerate_seg<false, true, true, NARROW> : k_enumerate_seg<false, true, false, NARROW>)
                      : (one ? k_enumerate_seg<false, false, true, NARROW>
                             : k_enumerate_seg<false, false, false, NARROW>));
}
}  // namespace

void launch_enumerate(dss_handle* h, int stbuf, int dst_list, int adv) {
  (void)adv;
  ListBuf& L = h->lb[dst_list];
  const Geo& g = h->g;
  prof_mark(h, 3);
  // FP32 cutoffs.  The electro-chemical range beats the pair-mean lubrication
  // cutoff for every pair when it beats the largest; only between the two do
  // both enter the candidate test.
  EnumCut q;
  const bool mean = g.mode == 0, wide = g.de > 0.0 && g.de >= g.delta * h->a_max;
  q.sc = mean && !wide ? 1.0f + 0.5f * (float)g.delta : 1.0f;
  q.sd = mean ? (wide ? (float)g.de : 0.0f) : (float)(g.delta * g.a0 > g.de ? g.delta * g.a0 : g.de);
  q.lc = mean ? 1.0f + 0.5f * (float)g.delta : 1.0f;
  q.ld = mean ? 0.0f : (float)(g.delta * g.a0);
  q.de = (float)g.de;
  const bool ech = g.de > 0.0 && mean && !wide;
  // with electro-chemical forces over cells of many particles (long ranges)
  // most listed pairs lie beyond the lubrication range: rows put the others
  // first, so that the pair kernel's warps meet runs of pairs without
  // lubrication (short rows gain less than the reordering costs)
  const bool split = g.de > 0.0 && !h->enum_walk && h->n >= 8 * (int64_t)g.ncell;
  const int tile = split ? 64 : 256;
  const RowSums R{h->row_sums, h->row_sums + h->row_tiles, split ? 6 : 8};
  const unsigned blocks = (unsigned)h->enum_blocks;
  if (h->enum_walk) {
    auto kw = g.nclass > 1 ? (ech ? k_enumerate_classes<true> : k_enumerate_classes<false>)
                           : (ech ? k_enumerate<true> : k_enumerate<false>);
    launch_dep(kw, blocks, kThreads, h->stream, g, h->ig, h->sg, h->st[stbuf], h->posf, h->cellid, h->cell_start, L, R,
               h->status, q);
  } else {
    const bool one = h->K == 1;
    auto ks = h->enum_narrow ? seg_kernel<true>(ech, split, one) : seg_kernel<false>(ech, split, one);
    launch_dep(ks, blocks, 32 * kRows, h->stream, g, h->ig_host[0], h->ig, h->sg, h->st[stbuf], h->posf, h->cellid,
                                             h->cell_start, L.list, L.count, h->offs, h->enum_inst, R, h->status, q);
  }
  prof_mark(h, 4);
  auto kr = split ? k_rows<true, 64> : k_rows<false, 256>;
  launch_dep(kr, ((int)h->n + tile - 1) / tile, kRowThreads, h->stream, (int)h->n, g.M, g.Ms, g.pcap, h->st[stbuf].id, L,
             h->offs, h->bw_count, h->cellid, h->cell_more, R, h->status);
  h->last_list = dst_list;
}
