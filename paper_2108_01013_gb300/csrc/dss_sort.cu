// Counting sort of the particles into cells (Sec. II A; the paper follows
// Hoetzlein's counting sort), redone every step with no Verlet skin:
//   1. predictor + Lees-Edwards wrap (Eq. 15a-b, 16) fused with the cell key,
//      a warp-aggregated histogram (one atomic per distinct key per warp) and
//      the ids of each cell's particles (a row of bcap places per cell);
//   2. exclusive scan of the histogram (from its tiles' sums, or by decoupled
//      look-back on large grids);
//   3. each particle finds its place (its cell's start plus its rank by id
//      among the cell's ids, so that the order is deterministic) and writes its
//      state there; the predicted position and velocity are those stored by
//      step 1 (SoA, source order).
// Particles move little in a step, so the writes of step 3 are nearly as
// coalesced as its reads; a scatter of indices before it and reads through
// them cost a kernel and two dependent loads more (20,000 spheres 45.7 -> 43.9
// us a step, 100,000 77.5 -> 76.6, 1M 474 -> 466).
#include <algorithm>

#include "dss_predict.cuh"

namespace {

constexpr int kThreads = 256;

// 1. key + warp-aggregated histogram; the last block sets the geometry
__global__ void __launch_bounds__(kThreads)
k_key_hist(const __grid_constant__ Geo g, const InstGeo* __restrict__ ig, const __grid_constant__ StateBuf s,
           DevStatus* st, bool predict, const __grid_constant__ SortOut q) {
  dep_wait();
  if (dev_err(st)) return;
  reset_scans(q);
  if (blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x == 0) {
      st->w[ST_MAXROW] = 0;
      st->w[ST_BAND] = 0;
      st->w[ST_NCONT] = 0;
    }
    set_step_geo(g, ig, st, predict ? 1 : 0, q.sg);
    return;
  }
  const int i = blockIdx.x * blockDim.x + threadIdx.x, n = g.n;
  if (i >= n) return;
  const InstGeo& I = ig[s.inst[i]];
  const int id = s.id[i], cls = s.cls[i];
  double x = s.x[i], y = s.x[n + i], z = s.x[2 * n + i];
  if (predict) {
    const Pred p = predict_one(g, I, st, 1, x, y, z, s.u[i], s.u[n + i], s.u[2 * n + i], s.al[i], s.al[n + i],
                               s.al[2 * n + i]);
    store_pred(q, n, i, p);
    x = p.x;
    y = p.y;
    z = p.z;
  }
  key_insert(q, i, cell_key(I, cls, x, y, z), id);
}

// The ids below mine among those beyond a full cell's row, in its chain of links
// (SortOut): a link is a round or more of loads for up to 32 ids, the next one on
// its way.  The work is the cell's own, quadratic in its particles as for every
// other cell.  20,000 small spheres segregated from the large ones, a thousand to
// a cell whose row holds 168: 59 us for the kernel (41 with all ids of a cell side
// by side, written by a kernel of its own that every step paid for).  A clump of
// 50,000 in a dilute box, rows of four: 10.3 us, a step 60 us from the first on.
// (Ranked over all particles' keys, with longer rows from the host's next call,
// the steps of the first call took 1380 us each.)
__device__ __noinline__ int rank_beyond_row(const int* __restrict__ id, int mine, int first, int left,
                                            const int* __restrict__ next, const unsigned* __restrict__ lanes) {
  int rank = 0, e = first;
  unsigned m = e ? lanes[e - 1] : 0u;
  int to = e ? next[e - 1] : 0;
  while (e && left > 0) {
    const int base = (e - 1) & ~31;
    unsigned cur = m;
    left -= __popc(cur);
    // the next link comes while this one's ids do
    e = to;
    m = e ? lanes[e - 1] : 0u;
    to = e ? next[e - 1] : 0;
    while (cur) {
      int v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        v[u] = cur ? id[base + __ffs(cur) - 1] : 0x7fffffff;
        cur &= cur - 1u;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) rank += v[u] < mine;
    }
  }
  return rank;
}

// 3. the place of each particle: inside a cell by id, so that the sorted order,
// and with it every summation order downstream, is a function of positions and
// ids alone; its state written there (WAVE: the wave of Eq. 17 is on, compiled
// out otherwise).
template <bool WAVE>
__global__ void __launch_bounds__(kThreads, 4)
k_rank_gather(Geo g, const InstGeo* __restrict__ ig, StateBuf src, StateBuf dst, const int* __restrict__ key,
              const int* __restrict__ cell_start, const int* __restrict__ cell_ids, int bcap,
              const int* __restrict__ more, const int* __restrict__ link_next,
              const unsigned* __restrict__ link_lanes, int* __restrict__ cell_count, int* __restrict__ tile_count,
              int clear, int* __restrict__ perm, int* __restrict__ cellid, float4* __restrict__ posf, DevStatus* st,
              int most_seg, int long_seg, bool predict, const double* __restrict__ pred,
              const signed char* __restrict__ xc) {
  dep_wait();
  if (dev_err(st)) return;
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = g.n;
  // the histogram of the next operation
  for (int t = o; t < clear; t += gridDim.x * blockDim.x) cell_count[t] = 0;
  if (clear)
    for (int t = o; t < kTileCopies * kScanTiles; t += gridDim.x * blockDim.x) tile_count[t] = 0;
  if (o >= n) return;
  const int k = key[o];
  const int id = src.id[o];
  const int inst = src.inst[o], iy = src.iy[o], cross = predict ? (int)xc[o] : 0;
  const unsigned char cls = src.cls[o];
  const double a = src.a[o];
  const int c0 = cell_start[k], cnt = cell_start[k + 1] - c0;
  // the state goes out with the loads that find its place
  Pred p;
  double wv3[3], wa[3];
  if (predict) {
    p.x = pred[o]; p.y = pred[n + o]; p.z = pred[2 * n + o];
    p.ux = pred[3 * n + o]; p.uy = pred[4 * n + o]; p.uz = pred[5 * n + o];
  } else {
    p.x = src.x[o]; p.y = src.x[n + o]; p.z = src.x[2 * n + o];
    p.ux = src.u[o]; p.uy = src.u[n + o]; p.uz = src.u[2 * n + o];
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    wv3[c] = src.w[c * n + o];
    wa[c] = src.aw[c * n + o];
  }
  int rank = 0;
  const int4* __restrict__ row = reinterpret_cast<const int4*>(cell_ids + (int64_t)k * bcap);
  const int held = min(cnt, bcap);
  for (int q = 0; q < held; q += 4) {
    const int4 v = __ldg(row + (q >> 2));
    rank += (v.x < id) + (q + 1 < held && v.y < id) + (q + 2 < held && v.z < id) + (q + 3 < held && v.w < id);
  }
  if (cnt > bcap) {
    rank += rank_beyond_row(src.id, id, more[k], cnt - bcap, link_next, link_lanes);
    if (rank == 0) st->w[ST_CELL] = 1;
  }
  // (the search's segments: a segment's cells lie among the most_seg from its
  // first particle's on)
  if (rank == 0 && cell_start[min(k + most_seg, g.ncell)] - c0 > long_seg) st->w[ST_LONG] = 1;
  const int f = c0 + rank;
  perm[f] = o;
  cellid[f] = k;
  const InstGeo& I = ig[inst];
  dst.x[f] = p.x; dst.x[n + f] = p.y; dst.x[2 * n + f] = p.z;
  dst.u[f] = p.ux; dst.u[n + f] = p.uy; dst.u[2 * n + f] = p.uz;
  if (predict) {
    const double hdt = g.hdt;
    if (g.precision == DSS_FP64)
      for (int c = 0; c < 3; ++c) wv3[c] = __dadd_rn(wv3[c], __dmul_rn(hdt, wa[c]));
    else
      for (int c = 0; c < 3; ++c) wv3[c] = __fma_rn(hdt, wa[c], wv3[c]);
  } else {
    for (int c = 0; c < 3; ++c) {
      dst.al[c * n + f] = src.al[c * n + o];
      dst.aw[c * n + f] = wa[c];
    }
  }
  for (int c = 0; c < 3; ++c) dst.w[c * n + f] = wv3[c];
  const double w0 = wv3[0], w1 = wv3[1], w2 = wv3[2];
  dst.a[f] = a;
  dst.id[f] = id;
  dst.inst[f] = inst;
  dst.cls[f] = cls;
  // image count: leaving through the top is one image up
  dst.iy[f] = iy - cross;
  // FP32 copies relative to the ambient flow for the FP32 pair arithmetic:
  // u - U_inf(x) and w - Omega_inf are O(gdot a), free of O(gdot L) terms
  Rec8 mv;
  if (WAVE) {
    // the wave of Eq. 17 at the centre, once per evaluation: its part of
    // U_inf,x and of the local rate dU_inf,x/dy
    double sn, cs;
    sincos(I.wave_k * p.y, &sn, &cs);
    const double ws = g.wave_amp * sn, wc = g.wave_amp * I.wave_k * cs;
    dst.wv[f] = make_double2(ws, wc);
    if (g.precision == DSS_MIXED) {
      dst.wvf[f] = make_float2(f32_rn(wc), f32_rn(ws));
      mv = Rec8{f32_rn(p.ux - I.gdot * p.y - ws), f32_rn(p.uy), f32_rn(p.uz), f32_rn(w0), f32_rn(w1),
                f32_rn(w2 + 0.5 * (I.gdot + wc))};
    }
  } else if (g.precision == DSS_MIXED) {
    mv = Rec8{f32_rn(p.ux - I.gdot * p.y), f32_rn(p.uy), f32_rn(p.uz), f32_rn(w0), f32_rn(w1),
              f32_rn(w2 + 0.5 * I.gdot)};
  }
  // cell-local position (FP32 for the enumeration prefilter; in mixed
  // precision also the low words, for double-float pair geometry)
  const int kl = (k - I.cell_base) % I.ncell_layer;
  int cx = kl % I.nc[0];
  int cy = (kl / I.nc[0]) % I.nc[1];
  int cz = kl / (I.nc[0] * I.nc[1]);
  const double lx = __fma_rn(-f64_of_nonneg(cx), I.cs[0], p.x),
               ly = __fma_rn(-f64_of_nonneg(cy), I.cs[1], p.y),
               lz = __fma_rn(-f64_of_nonneg(cz), I.cs[2], p.z);
  // the FP32 words and (mixed precision) the low words of the double-float
  // pair geometry
  float4 pf, pl;
  f32_split(lx, pf.x, pl.x);
  f32_split(ly, pf.y, pl.y);
  f32_split(lz, pf.z, pl.z);
  f32_split(a, pf.w, pl.w);
  posf[f] = pf;
  if (g.precision == DSS_MIXED) {
    mv.v[6] = __int_as_float(cx | (cy << 10) | (cz << 20));
    mv.v[7] = __int_as_float(id);
    store_rec(dst.rec + rec_geometry(f), Rec8{pf.x, pf.y, pf.z, pf.w, pl.x, pl.y, pl.z, pl.w});
    store_rec(dst.rec + rec_motion(f), mv);
  }
}

}  // namespace

// Single-pass exclusive scan with decoupled look-back.  Tiles are taken in
// launch order through an atomic ticket, so every predecessor a tile waits
// on is already running; each wait is bounded and reports DSS_ERR_TIMEOUT.
namespace {
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
static_assert(kScanTile == kScanThreads * kScanItems, "a thread scans eight bins");

__host__ __device__ constexpr int scan_pad(int q) { return q + (q >> 5); }   // no bank conflicts

// A tile is loaded and stored coalesced through shared memory; each thread
// scans 8 consecutive items of it.  The input is cleared as soon as it is
// read when zero_in is set (the histogram of the next operation).
__global__ void __launch_bounds__(kScanThreads)
k_scan(const int* __restrict__ in, int* __restrict__ out, int count,
       unsigned long long* status, int* ticket, DevStatus* st, int zero_in) {
  dep_wait();
  __shared__ int s_tile, s_err, s_prefix, s_agg;
  __shared__ int s_warp[kScanThreads / 32];
  __shared__ int s_v[scan_pad(kScanTile)];
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1);
  if (threadIdx.x == 32) s_err = dev_err(st);
  __syncthreads();
  if (s_err) return;
  const int tile = s_tile;
  const int base = tile * kScanTile;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const int q = k * kScanThreads + threadIdx.x;
    const int idx = base + q;
    int x = 0;
    if (idx < count) {
      x = in[idx];
      if (zero_in) const_cast<int*>(in)[idx] = 0;
    }
    s_v[scan_pad(q)] = x;
  }
  __syncthreads();
  int v[kScanItems];
  int local = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    v[k] = s_v[scan_pad(threadIdx.x * kScanItems + k)];
    local += v[k];
  }
  // block exclusive scan of the per-thread sums
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = local;
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    const int w = lane < kScanThreads / 32 ? s_warp[lane] : 0;
    int wi = w;
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, wi, d);
      if (lane >= d) wi += t;
    }
    if (lane < kScanThreads / 32) s_warp[lane] = wi - w;   // exclusive warp offsets
    if (lane == kScanThreads / 32 - 1) s_agg = wi;
  }
  __syncthreads();
  // tile prefix by look-back (warp 0) while every thread stores its
  // tile-local exclusive values
  if (wid == 0) {
    const int agg = s_agg;
    const int prefix = lookback_warp(status, tile, agg, st);
    if (lane == 0) {
      s_prefix = prefix;
      if (base + kScanTile >= count) out[count] = prefix + agg;   // total
    }
  }
  int run = incl - local + s_warp[wid];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    s_v[scan_pad(threadIdx.x * kScanItems + k)] = run;
    run += v[k];
  }
  __syncthreads();
  const int pre = s_prefix;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const int q = k * kScanThreads + threadIdx.x;
    const int idx = base + q;
    if (idx < count) out[idx] = s_v[scan_pad(q)] + pre;
  }
}
}  // namespace

// The same for grids of up to kScanTiles tiles, whose sums the histogram kept: a
// tile's first bin is the sum of the tiles before it, so that no block waits
// for another: one round of loads and one barrier.  The look-back of k_scan took 2
// us more (8.2 -> 6.2 at 20k and 100k, 10.3 -> 8.0 at 140k bins, 12.1 -> 8.1 at
// 314k); a thread sums one tile's copies, so that 256 tiles are the limit.
// The counts stay for the ranking kernel to clear.
namespace {
__global__ void __launch_bounds__(kScanThreads)
k_scan_tiles(const int* __restrict__ in, const int* __restrict__ tile_count, int* __restrict__ out, int count,
             const DevStatus* st) {
  __shared__ int s_warp[kScanThreads / 32], s_before[kScanThreads / 32];
  dep_wait();
  if (dev_err(st)) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, tile = blockIdx.x;
  const int i = tile * kScanTile + threadIdx.x * kScanItems;
  int v[kScanItems];
  if (i + kScanItems <= count) {
    const int4 a = *reinterpret_cast<const int4*>(in + i), b = *reinterpret_cast<const int4*>(in + i + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) v[k] = i + k < count ? in[i + k] : 0;
  }
  {
    const int t = threadIdx.x % kScanTiles;
    int sum = 0;
    if (t < tile) {
#pragma unroll
      for (int c = threadIdx.x / kScanTiles; c < kTileCopies; c += kScanThreads / kScanTiles)
        sum += tile_count[c * kScanTiles + t];
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) s_before[wid] = sum;
  }
  int local = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) local += v[k];
  int incl = local;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  int run = incl - local;
#pragma unroll
  for (int w = 0; w < kScanThreads / 32; ++w) run += s_before[w] + (w < wid ? s_warp[w] : 0);
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    const int t = v[k];
    v[k] = run;
    run += t;
  }
  if (i + kScanItems <= count) {
    *reinterpret_cast<int4*>(out + i) = make_int4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<int4*>(out + i + 4) = make_int4(v[4], v[5], v[6], v[7]);
    if (i + kScanItems == count) out[count] = run;
  } else {
#pragma unroll
    for (int k = 0; k < kScanItems; ++k)
      if (i + k < count) {
        out[i + k] = v[k];
        if (i + k + 1 == count) out[count] = k + 1 < kScanItems ? v[k + 1] : run;
      }
  }
}
}  // namespace

int scan_tiles_for(int count) { return (count + kScanTile - 1) / kScanTile; }

// The cells' starts from their counts.
static void launch_cell_scan(dss_handle* h) {
  const int count = h->g.ncell, tiles = std::max(scan_tiles_for(count), 1);
  if (tiles <= kScanTiles)
    launch_dep(k_scan_tiles, tiles, kScanThreads, h->stream, h->cell_count, h->tile_count, h->cell_start, count,
               h->status);
  else
    launch_dep(k_scan, tiles, kScanThreads, h->stream, h->cell_count, h->cell_start, count, h->scan_status,
               h->scan_ticket, h->status, 1);
}

void launch_sort(dss_handle* h, bool predict, int src, int dst, bool keyed) {
  const int n = (int)h->n;
  const int blocks = (n + kThreads - 1) / kThreads;
  prof_mark(h, 0);
  if (!keyed) launch_dep(k_key_hist, blocks + 1, kThreads, h->stream, h->g, h->ig, h->st[src], h->status, predict, sort_out(h));
  prof_mark(h, 1);
  launch_cell_scan(h);
  prof_mark(h, 2);
  const int clear = scan_tiles_for(h->g.ncell) <= kScanTiles ? h->g.ncell : 0;
  const SortOut so = sort_out(h);
  auto k = h->g.wave ? k_rank_gather<true> : k_rank_gather<false>;
  launch_dep(k, blocks, kThreads, h->stream, h->g, h->ig, h->st[src], h->st[dst], h->key, h->cell_start, h->cell_ids,
             h->cell_cap, so.more, so.link_next, so.link_lanes, h->cell_count, h->tile_count, clear, h->perm, h->cellid,
             h->posf, h->status, h->enum_most_seg, h->enum_long_seg, predict, h->pred, h->xc);
}

// Self-test of the integer-operation conversions (f32_rn, f32_split, f64_of,
// floor_mul, f64_of_nonneg) over caller-chosen inputs.
namespace {
__global__ void k_selftest_conversions(const double* __restrict__ v, int64_t n, double inv, float invf,
                                       float* __restrict__ hi, float* __restrict__ shi,
                                       float* __restrict__ slo, double* __restrict__ back,
                                       int* __restrict__ fl, const int* __restrict__ ci,
                                       double* __restrict__ cd) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const double x = v[k];
    const float h = f32_rn(x);
    hi[k] = h;
    f32_split(x, shi[k], slo[k]);
    back[k] = f64_of(h);
    fl[k] = floor_mul(x, inv, invf);
    cd[k] = f64_of_nonneg(ci[k]);
  }
}
}  // namespace

extern "C" int dss_selftest_conversions(const double* v, int64_t n, double inv, float* hi, float* split_hi,
                                        float* split_lo, double* back, int32_t* floor_out,
                                        const int32_t* ints, double* ints_out, void* cuda_stream) {
  if (n < 0 || (n > 0 && (!v || !hi || !split_hi || !split_lo || !back || !floor_out || !ints || !ints_out)))
    return DSS_ERR_ARG;
  if (n == 0) return DSS_OK;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  k_selftest_conversions<<<(int)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096), 256, 0, s>>>(
      v, n, inv, (float)inv, hi, split_hi, split_lo, back, floor_out, ints, ints_out);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) return DSS_ERR_CUDA;
  return DSS_OK;
}
