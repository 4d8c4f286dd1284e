// lgs_bin.cu -- preprocess, angular-tile binning, per-tile depth sort.
//
// Pipeline of one lgs_bin_sort (all on the caller's stream, no host sync):
//   k_tables      per frame: binary32 sine / direction tables of the tile
//                 rows and columns (pixel-centre extremes of each tile)
//   k_preprocess  per (frame, surfel) item: 64 B compositing record, pixel
//                 box, depth key = bits of binary32 |mu_sensor|; the item's
//                 tiles (a range of tile rows times a circular range of tile
//                 columns, stored per item) and one count per covered tile
//                 (shared-memory counters per CTA, one atomic per tile)
//   k_tile_scan   one CTA: exclusive scan of the tile counts -> every tile's
//                 [start, end) and its fill cursor; capacity check; the
//                 longest-first tile order of the persistent kernels; the
//                 list of tiles longer than kLongList
//   k_emit        every item appends (depth key << 32 | item) to the bucket
//                 of each tile of its stored set (order inside a bucket
//                 arbitrary)
//   k_long_split  buckets of more than 2048 keys: partitioned by depth into
//                 groups of about 1024 keys, one CTA per bucket, longest first
//   k_tile_sort   sort every shorter bucket and every group by the 64-bit key,
//                 one CTA each (in sparse calls a warp each of the shortest), by
//                 distribution in shared memory; write the item list
// The result is the order of the key (tile, depth, item): per tile, by depth,
// ties by item index.
#include <cuda_runtime.h>

#include "lgs_internal.cuh"

namespace lgs {

// ---------------------------------------------------------------------------
// Descriptors and tables
// ---------------------------------------------------------------------------
__global__ void k_write_desc(const __grid_constant__ Desc h, Desc* __restrict__ d) {
  const int nw = static_cast<int>(sizeof(Desc) / 4);
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&h);
  uint32_t* dst = reinterpret_cast<uint32_t*>(d);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nw; i += gridDim.x * blockDim.x) dst[i] = src[i];
}

cudaError_t launch_write_desc(const Desc& h, Desc* d, Status*, cudaStream_t s) {
  k_write_desc<<<4, 256, 0, s>>>(h, d);
  return cudaGetLastError();
}

__global__ void k_tables(const Desc* __restrict__ D, float* __restrict__ tab, Status* __restrict__ st,
                         uint32_t* __restrict__ loss_acc, uint32_t loss_words, uint32_t* __restrict__ tcount,
                         uint32_t n_tiles) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  const FrameDev& F = D->f[blockIdx.x];
  // the tile counts start at zero (k_preprocess adds into them)
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_tiles; i += gridDim.x * blockDim.x) tcount[i] = 0u;
  // the loss accumulators start every binning at zero
  if (blockIdx.x == 0)
    for (uint32_t i = threadIdx.x; i < loss_words; i += blockDim.x) loss_acc[i] = 0u;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->required_pairs = 0;
    st->n_pairs = 0;
    st->n_vis = 0;
    st->overflow = 0;
    st->timeout = 0;
    st->check = 0;
    st->work_counter = 0;
    st->work_counter2 = 0;
    for (int c = 0; c < kBwdClasses; ++c) st->bq_count[c] = 0;
    st->evals_fwd = 0;
    st->evals_bwd = 0;
    st->contrib_fwd = 0;
    st->contrib_bwd = 0;
    st->alg_fwd = 0;
    st->loss_ticket = 0;
    st->count_ticket = 0;
    st->n_long = 0;
    st->n_segs = 0;
    st->seg_counter = 0;
    st->seg_done = 0;
    st->n_big = 0;
    st->long_sort_counter = 0;
    st->n_groups = 0;
    st->long_counter_fwd = 0;
    st->long_counter_bwd = 0;
    st->long_done_fwd = 0;
    st->long_done_bwd = 0;
  }
  for (int i = threadIdx.x; i < F.ntr; i += blockDim.x) {
    const int r0 = i * F.th;
    const int r1 = ((i + 1) * F.th < F.H ? (i + 1) * F.th : F.H) - 1;
    tab[F.row_tab + 2 * i] = bin_sin(bin_row_elev(r0, F.H, F.emin, F.emax));
    tab[F.row_tab + 2 * i + 1] = bin_sin(bin_row_elev(r1, F.H, F.emin, F.emax));
  }
  for (int j = threadIdx.x; j < F.ntc; j += blockDim.x) {
    const int c0 = j * F.tw;
    const int c1 = ((j + 1) * F.tw < F.W ? (j + 1) * F.tw : F.W) - 1;
    float cs, sn;
    bin_col_dir(c0, F.W, cs, sn);
    tab[F.col_tab + 4 * j] = cs;
    tab[F.col_tab + 4 * j + 1] = sn;
    bin_col_dir(c1, F.W, cs, sn);
    tab[F.col_tab + 4 * j + 2] = cs;
    tab[F.col_tab + 4 * j + 3] = sn;
  }
}

// Calls fn(global tile id) for every tile the item's bounding cone meets:
// rows ascending, then the candidate column ranges of bin_col_window in order.
// Only the tile rows that hold a pixel row of the item's pixel box (which
// pads the cone's elevation band by a whole pixel row on each side) are
// tested: a tile row the cone meets always holds one.
template <class Fn>
__device__ __forceinline__ uint32_t for_each_tile(const BinGeom& g, const FrameDev& F, const float* __restrict__ tab,
                                                  const float4& pbox, Fn fn) {
  const float4* ct = reinterpret_cast<const float4*>(tab + F.col_tab);
  ColWin w;
  bin_col_window(g, F, w);
  int ra = 0, rb = F.ntr - 1;
  if (!g.all_rows) {
    ra = max(0, static_cast<int>(pbox.x) / F.th);
    rb = min(F.ntr - 1, static_cast<int>(pbox.y) / F.th);
  }
  uint32_t n = 0;
  for (int r = ra; r <= rb; ++r) {
    if (!bin_row_hit(g, tab[F.row_tab + 2 * r], tab[F.row_tab + 2 * r + 1])) continue;
    const uint32_t rowbase = F.tile_base + static_cast<uint32_t>(r * F.ntc);
    for (int pass = 0; pass < 2; ++pass) {
      const int ja = pass ? w.b0 : w.a0, jb = pass ? w.b1 : w.a1;
      for (int jc = ja; jc <= jb; ++jc) {
        if (!bin_col_hit(g, ct[jc])) continue;
        fn(rowbase + static_cast<uint32_t>(jc));
        ++n;
      }
    }
  }
  return n;
}

// The tiles an item's bounding cone meets form a product of tile rows and
// tile columns (the row test depends on the row only, the column test on
// the column only).  The passing rows form one range and the passing columns
// one circular range (the cone is convex in elevation and in azimuth, and a
// tile between two passing tiles lies deep inside the cone), so an item's
// tiles are stored as rows [r0, r1] and nc columns from c0 on, modulo the
// column count.  Should the passing rows or columns not form one range (a
// decision at the binary32 edge of the cone), tile_set returns false and the
// caller enumerates the tiles one by one instead (for_each_tile).
struct TileSet {
  int r0, r1, c0, nc;
};

constexpr uint32_t kTsEnumerate = 0xffffffffu;   // stored tile set: enumerate tile by tile

__device__ __forceinline__ bool tile_set(const BinGeom& g, const FrameDev& F, const float* __restrict__ tab,
                                         const float4& pbox, TileSet& t) {
  const float4* ct = reinterpret_cast<const float4*>(tab + F.col_tab);
  t.r0 = 0;
  t.r1 = -1;
  t.c0 = 0;
  t.nc = 0;
  if (F.ntr >= 0xffff || F.ntc >= 0xffff) return false;
  int ra = 0, rb = F.ntr - 1;
  if (!g.all_rows) {
    ra = max(0, static_cast<int>(pbox.x) / F.th);
    rb = min(F.ntr - 1, static_cast<int>(pbox.y) / F.th);
  }
  int r0 = -1, r1 = -1, nr = 0;
  for (int r = ra; r <= rb; ++r) {
    if (!bin_row_hit(g, tab[F.row_tab + 2 * r], tab[F.row_tab + 2 * r + 1])) continue;
    if (r0 < 0) r0 = r;
    r1 = r;
    ++nr;
  }
  if (nr == 0) return true;
  if (nr != r1 - r0 + 1) return false;
  ColWin w;
  bin_col_window(g, F, w);
  // the candidate columns in circular order (the window's second range
  // continues the first across the azimuth seam)
  int prev = -1, runs = 0, first = 0, second = 0, n = 0;
  for (int pass = 0; pass < 2; ++pass) {
    const int ja = pass ? w.b0 : w.a0, jb = pass ? w.b1 : w.a1;
    for (int jc = ja; jc <= jb; ++jc) {
      if (!bin_col_hit(g, ct[jc])) continue;
      if (prev < 0 || jc != (prev + 1 == F.ntc ? 0 : prev + 1)) {
        ++runs;
        if (runs == 1) first = jc;
        else second = jc;
      }
      prev = jc;
      ++n;
    }
  }
  if (n == 0) return true;
  if (runs == 1) {
    t.c0 = first;
  } else if (runs == 2 && first == 0 && prev == F.ntc - 1) {
    t.c0 = second;        // one range across the seam, seen from column 0
  } else {
    return false;
  }
  t.r0 = r0;
  t.r1 = r1;
  t.nc = n;
  return true;
}

template <class Fn>
__device__ __forceinline__ void for_each_in_set(const TileSet& t, const FrameDev& F, Fn fn) {
  for (int r = t.r0; r <= t.r1; ++r) {
    const uint32_t rowbase = F.tile_base + static_cast<uint32_t>(r * F.ntc);
    for (int k = 0; k < t.nc; ++k) {
      int jc = t.c0 + k;
      if (jc >= F.ntc) jc -= F.ntc;
      fn(rowbase + static_cast<uint32_t>(jc));
    }
  }
}

// A lane's tile set within the warp: its first row's tile 0 and the frame's
// column count with it (a warp's items may lie in two frames).
struct WarpSet {
  uint32_t row0, ntc;   // global id of tile (r0, 0); columns of the frame
  int nr, c0, nc;
};

__device__ __forceinline__ WarpSet warp_set(const TileSet& t, const FrameDev& F) {
  return WarpSet{F.tile_base + static_cast<uint32_t>(t.r0 * F.ntc), static_cast<uint32_t>(F.ntc), t.r1 - t.r0 + 1, t.c0,
                 t.nc};
}

// Calls fn(tile) for every tile of every lane's set; all lanes call it.  A set
// of up to kOwnTiles tiles is walked by its lane, a larger one by the whole
// warp: a surfel beside the sensor meets hundreds of tiles, and its CTA waited
// for its lane (8 keyframes of a 1M map: the kernel 744 -> 603 us; a street
// frame, 200k surfels, and six batched maps as before, 21 and 272 us).  Line at
// 8: 642, 26 and 381 us (the warp takes the sets in turn, with a broadcast each);
// 20: 612, 21.6, 272; 64: 596, 22.6, 273.  Several items per thread were worse
// (1.41 ms at 6): the near surfels are neighbours in the map, so they come to
// the same CTAs.
constexpr int kOwnTiles = 32;

template <class Fn>
__device__ __forceinline__ void for_warp_sets(const WarpSet& w, int lane, Fn fn) {
  const int n = w.nr * w.nc;
  if (n > 0 && n <= kOwnTiles) {
    for (int r = 0; r < w.nr; ++r)
      for (int k = 0; k < w.nc; ++k) {
        uint32_t jc = static_cast<uint32_t>(w.c0 + k);
        if (jc >= w.ntc) jc -= w.ntc;
        fn(w.row0 + static_cast<uint32_t>(r) * w.ntc + jc);
      }
  }
  for (uint32_t big = __ballot_sync(0xffffffffu, n > kOwnTiles); big; big &= big - 1) {
    const int l = __ffs(big) - 1;
    const uint32_t row0 = __shfl_sync(0xffffffffu, w.row0, l), ntc = __shfl_sync(0xffffffffu, w.ntc, l);
    const uint32_t c0 = __shfl_sync(0xffffffffu, static_cast<uint32_t>(w.c0), l);
    const uint32_t nc = __shfl_sync(0xffffffffu, static_cast<uint32_t>(w.nc), l);
    const uint32_t m = __shfl_sync(0xffffffffu, static_cast<uint32_t>(n), l);
    for (uint32_t i = lane; i < m; i += 32) {
      const uint32_t r = i / nc;
      uint32_t jc = c0 + (i - r * nc);
      if (jc >= ntc) jc -= ntc;
      fn(row0 + r * ntc + jc);
    }
  }
}

__device__ __forceinline__ uint2 pack_set(const TileSet& t) {
  return make_uint2(static_cast<uint32_t>(t.r0) | (static_cast<uint32_t>(t.r1 < 0 ? 0 : t.r1) << 16),
                    static_cast<uint32_t>(t.c0) | (static_cast<uint32_t>(t.nc) << 16));
}

__device__ __forceinline__ TileSet unpack_set(uint2 p) {
  TileSet t;
  t.r0 = static_cast<int>(p.x & 0xffffu);
  t.r1 = static_cast<int>(p.x >> 16);
  t.c0 = static_cast<int>(p.y & 0xffffu);
  t.nc = static_cast<int>(p.y >> 16);
  return t;
}

// Per-CTA tile counters in shared memory: when all of a CTA's items belong
// to one frame with at most kAggTiles tiles, its per-tile atomics go to
// shared memory and each tile it touched gets one global atomic (items are
// usually stored in scan order, so a CTA touches few tiles).
constexpr int kAggTiles = 4096;

struct AggWin {
  bool local;
  uint32_t base, n;   // global id of the frame's tile 0, tiles of the frame
};

__device__ __forceinline__ AggWin agg_window(const Desc& D) {
  const int64_t first = static_cast<int64_t>(blockIdx.x) * blockDim.x;
  int64_t last = first + blockDim.x - 1;
  if (last >= D.n_items) last = D.n_items - 1;
  AggWin a;
  a.local = false;
  a.base = 0;
  a.n = 0;
  if (first > last) return a;
  const int f0 = frame_of_item(D, first), f1 = frame_of_item(D, last);
  const FrameDev& F = D.f[f0];
  a.n = static_cast<uint32_t>(F.ntr * F.ntc);
  a.base = F.tile_base;
  a.local = f0 == f1 && a.n <= static_cast<uint32_t>(kAggTiles);
  return a;
}

// ---------------------------------------------------------------------------
// Preprocess: record + key + box per (frame, surfel) item; tile counts
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_preprocess(const Desc* __restrict__ D, const float* __restrict__ tab,
                                                     float4* __restrict__ rec, float4* __restrict__ box,
                                                     uint32_t* __restrict__ key, uint32_t* __restrict__ cnt,
                                                     uint2* __restrict__ tset, uint32_t* __restrict__ tcount,
                                                     Status* __restrict__ st) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ uint32_t s_cnt[kAggTiles];
  const int64_t item = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool live = item < D->n_items;
  const AggWin aw = agg_window(*D);
  if (aw.local) {
    for (uint32_t t = threadIdx.x; t < aw.n; t += blockDim.x) s_cnt[t] = 0u;
    __syncthreads();
  }
  uint32_t c = 0;
  WarpSet ws{0u, 1u, 0, 0, 0};
  const auto count = [&](uint32_t t) {
    if (aw.local) atomicAdd(s_cnt + (t - aw.base), 1u);
    else atomicAdd(tcount + t, 1u);
  };
  if (live) {
    const int f = frame_of_item(*D, item);
    const FrameDev& F = D->f[f];
    const MapDev& M = D->m[F.map];
    const int64_t i = item - F.item_base;
    // every parameter load issued up front (the atomics below would otherwise
    // keep the compiler from hoisting them)
    const float4 q = reinterpret_cast<const float4*>(M.quat)[i];
    const float ls0 = M.ls[2 * i], ls1 = M.ls[2 * i + 1], lg = M.logit[i];
    BinGeom g;
    bin_geom(M.mean + 3 * i, M.ls + 2 * i, F, g);
    key[item] = __float_as_uint(g.r);
    const float4 pb = pixel_box(g, F);
    TileSet ts;
    if (tile_set(g, F, tab, pb, ts)) {
      ws = warp_set(ts, F);
      c = static_cast<uint32_t>((ts.r1 - ts.r0 + 1) * ts.nc);
      tset[item] = pack_set(ts);
    } else {
      c = for_each_tile(g, F, tab, pb, count);
      tset[item] = make_uint2(kTsEnumerate, kTsEnumerate);
    }
    cnt[item] = c;

    // compositing record (accuracy only): rotation of the unit quaternion,
    // axes to the sensor frame, activations
    const float inv = rsqrtf(q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w);
    const float w = q.x * inv, x = q.y * inv, y = q.z * inv, z = q.w * inv;
    // world-frame columns of R(q)
    const float c0x = 1.f - 2.f * (y * y + z * z), c0y = 2.f * (x * y + w * z), c0z = 2.f * (x * z - w * y);
    const float c1x = 2.f * (x * y - w * z), c1y = 1.f - 2.f * (x * x + z * z), c1z = 2.f * (y * z + w * x);
    const float c2x = 2.f * (x * z + w * y), c2y = 2.f * (y * z - w * x), c2z = 1.f - 2.f * (x * x + y * y);
    const float* R = F.R;
    // sensor frame: v_s = R^T v_w
    const float tux = R[0] * c0x + R[3] * c0y + R[6] * c0z, tuy = R[1] * c0x + R[4] * c0y + R[7] * c0z,
                tuz = R[2] * c0x + R[5] * c0y + R[8] * c0z;
    const float tvx = R[0] * c1x + R[3] * c1y + R[6] * c1z, tvy = R[1] * c1x + R[4] * c1y + R[7] * c1z,
                tvz = R[2] * c1x + R[5] * c1y + R[8] * c1z;
    const float nx = R[0] * c2x + R[3] * c2y + R[6] * c2z, ny = R[1] * c2x + R[4] * c2y + R[7] * c2z,
                nz = R[2] * c2x + R[5] * c2y + R[8] * c2z;
    const float isu = expf(-ls0), isv = expf(-ls1);
    const float alpha = 1.0f / (1.0f + expf(-lg));
    const float mx = g.x, my = g.y, mz = g.z;
    float4* out = rec + 4 * item;
    out[0] = make_float4(nx, ny, nz, nx * mx + ny * my + nz * mz);
    out[1] = make_float4(tux * isu, tuy * isu, tuz * isu, (tux * mx + tuy * my + tuz * mz) * isu);
    out[2] = make_float4(tvx * isv, tvy * isv, tvz * isv, (tvx * mx + tvy * my + tvz * mz) * isv);
    const float su = expf(ls0), sv = expf(ls1);
    out[3] = make_float4(alpha, su, sv, 0.f);
    box[item] = cull_box(g, F, pb, tux, tuy, tuz, tvx, tvy, tvz, su, sv);
  }
  __syncwarp();
  for_warp_sets(ws, threadIdx.x & 31, count);
  // visible-item count, one atomic per warp
  const uint32_t vis = __ballot_sync(0xffffffffu, c > 0);
  if ((threadIdx.x & 31) == 0 && vis) atomicAdd(&st->n_vis, static_cast<unsigned int>(__popc(vis)));
  if (aw.local) {
    __syncthreads();
    for (uint32_t t = threadIdx.x; t < aw.n; t += blockDim.x)
      if (s_cnt[t]) atomicAdd(tcount + aw.base + t, s_cnt[t]);
  }
}

// ---------------------------------------------------------------------------
// Tile offsets: one CTA scans the tile counts
// ---------------------------------------------------------------------------
constexpr int kScanCta = 1024;

constexpr uint32_t kLenCache = 4096;   // tiles whose list length the scan keeps in shared memory

// Bucket of a tile list length for the longest-first order: floor(log2(n)) + 1
// (0 for an empty tile), reversed so that bucket 0 holds the longest lists.
// Buckets of up to kSortMax keys are sorted in shared memory by one CTA;
// longer ones split into groups first (k_long_split), in this longest-first
// order.
constexpr uint32_t kSortMax = 2048;
// Buckets of up to kWarpSort keys are sorted by one warp.
constexpr uint32_t kWarpSort = 64;
constexpr int kOrderBuckets = 33;
__device__ __forceinline__ int order_bucket(uint32_t n) { return kOrderBuckets - 1 - (n ? 32 - __clz(n) : 0); }

__global__ void __launch_bounds__(kScanCta) k_tile_scan(uint32_t* __restrict__ tcur, uint32_t n_tiles,
                                                          uint2* __restrict__ ranges, Status* __restrict__ st,
                                                          int64_t cap, uint32_t* __restrict__ order,
                                                          uint32_t* __restrict__ longt, uint32_t* __restrict__ cbase) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ unsigned long long s_w[32];
  __shared__ uint32_t s_wc[32];
  __shared__ unsigned long long s_carry, s_tot;
  __shared__ uint32_t s_ccarry, s_ctot;
  __shared__ uint32_t s_bucket[kOrderBuckets];
  __shared__ uint32_t s_len[kLenCache];   // list lengths of the first tiles, kept for the order passes
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) {
    s_carry = 0;
    s_ccarry = 0;
  }
  if (tid < kOrderBuckets) s_bucket[tid] = 0;
  __syncthreads();
  for (uint32_t b0 = 0; b0 < n_tiles; b0 += kScanCta) {
    const uint32_t t = b0 + tid;
    const unsigned long long x = t < n_tiles ? tcur[t] : 0ull;
    // backward chunks of the list: ceil(n / kChunk)
    const uint32_t xc = static_cast<uint32_t>((x + kChunk - 1) / kChunk);
    unsigned long long v = x;
    uint32_t vc = xc;
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, v, o);
      const uint32_t yc = __shfl_up_sync(0xffffffffu, vc, o);
      if (lane >= o) {
        v += y;
        vc += yc;
      }
    }
    if (lane == 31) {
      s_w[wid] = v;
      s_wc[wid] = vc;
    }
    __syncthreads();
    // warp 0 turns the 32 warp totals into exclusive prefixes and the pass total
    if (wid == 0) {
      const unsigned long long x0 = s_w[lane];
      const uint32_t c0 = s_wc[lane];
      unsigned long long y = x0;
      uint32_t yc = c0;
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long z = __shfl_up_sync(0xffffffffu, y, o);
        const uint32_t zc = __shfl_up_sync(0xffffffffu, yc, o);
        if (lane >= o) {
          y += z;
          yc += zc;
        }
      }
      s_w[lane] = y - x0;
      s_wc[lane] = yc - c0;
      if (lane == 31) {
        s_tot = y;
        s_ctot = yc;
      }
    }
    __syncthreads();
    const unsigned long long wpre = s_w[wid], tot = s_tot;
    const uint32_t cpre = s_wc[wid], ctot = s_ctot;
    const unsigned long long start = s_carry + wpre + v - x;
    if (t < n_tiles) {
      // offsets past the capacity are never used: the emission is skipped
      const uint32_t s32 = static_cast<uint32_t>(start);
      if (t < kLenCache) s_len[t] = static_cast<uint32_t>(x);
      tcur[t] = s32;
      ranges[t] = x ? make_uint2(s32, static_cast<uint32_t>(start + x)) : make_uint2(0u, 0u);   // empty: (0, 0)
      // first chunk of the tile (non-decreasing over tiles: the chunk of a
      // global chunk index is found by binary search)
      cbase[t] = s_ccarry + cpre + vc - xc;
    }
    __syncthreads();
    if (tid == 0) {
      s_carry += tot;
      s_ccarry += ctot;
    }
    __syncthreads();
  }
  const unsigned long long total = s_carry;
  const bool over = total > static_cast<unsigned long long>(cap);
  if (tid == 0) {
    st->required_pairs = total;
    st->overflow = over ? 1u : 0u;
    st->n_pairs = over ? 0ull : total;
    st->n_chunks = over ? 0u : s_ccarry;   // at most pairs / kChunk + tiles
  }
  if (over) {
    // nothing is emitted: every tile renders empty
    for (uint32_t t = tid; t < n_tiles; t += kScanCta) ranges[t] = make_uint2(0u, 0u);
  }
  // work order of the persistent kernels: tiles by list length, longest
  // power-of-two class first (order inside a class is arbitrary; results do
  // not depend on it).  Both passes read the final ranges.
  __syncthreads();
  // one shared atomic per distinct class in a warp (most tiles of a frame
  // fall in a few classes, so per-tile atomics would serialise)
  // list length of tile t as the ranges now hold it
  const auto tile_len = [&](uint32_t t) -> uint32_t {
    if (over) return 0u;
    if (t < kLenCache) return s_len[t];
    const uint2 rg = ranges[t];
    return rg.y - rg.x;
  };
  for (uint32_t b0 = 0; b0 < n_tiles; b0 += kScanCta) {
    const uint32_t t = b0 + tid;
    const int b = t < n_tiles ? order_bucket(tile_len(t)) : -1;
    const uint32_t peers = __match_any_sync(0xffffffffu, b);
    if (b >= 0 && lane == __ffs(peers) - 1) atomicAdd(&s_bucket[b], static_cast<uint32_t>(__popc(peers)));
  }
  __syncthreads();
  // exclusive prefix of the 33 class counts by one warp (class 32 after the
  // other 32)
  static_assert(kOrderBuckets == 33, "one class per lane plus the last");
  if (wid == 0) {
    const uint32_t c = s_bucket[lane];
    uint32_t y = c;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    s_bucket[lane] = y - c;
    if (lane == 31) s_bucket[32] = y;
  }
  __syncthreads();
  for (uint32_t b0 = 0; b0 < n_tiles; b0 += kScanCta) {
    const uint32_t t = b0 + tid;
    const uint32_t len = t < n_tiles ? tile_len(t) : 0u;
    const int b = t < n_tiles ? order_bucket(len) : -1;
    const uint32_t peers = __match_any_sync(0xffffffffu, b);
    const int leader = __ffs(peers) - 1;
    uint32_t pos = 0;
    if (b >= 0 && lane == leader) pos = atomicAdd(&s_bucket[b], static_cast<uint32_t>(__popc(peers)));
    pos = __shfl_sync(0xffffffffu, pos, leader) + __popc(peers & ((1u << lane) - 1u));
    if (b >= 0) order[pos] = t;
    if (len > kLongList) longt[atomicAdd(&st->n_long, 1u)] = t;
    // k_long_split's buckets (found through the order)
    if (len > kSortMax) atomicAdd(&st->n_big, 1u);
  }
}

// ---------------------------------------------------------------------------
// Emission into the tile buckets
// ---------------------------------------------------------------------------
// Bound by the latency of its dependent steps (set, shared counter, run,
// 8-byte scattered store) and the CTA's three barriers.  One shared array, whose
// counters become the runs' next slots, instead of counters and bases: 16 KB
// less per CTA and one access less per pair; 8 keyframes of a 1M map 577 -> 517
// us, six batched maps 291 -> 279, a street frame (200k surfels) 13.7 -> 13.9.
// Large sets stay with their lanes here (by the whole warp 633, 282 and 14.4
// us: the fill is held up by its stores, not by the enumeration); several
// items per thread 570 to 635 us, CTAs of 128 and 512 threads 544 and 598.
__global__ void __launch_bounds__(256) k_emit(const Desc* __restrict__ D, const float* __restrict__ tab,
                                               const uint32_t* __restrict__ key, const uint32_t* __restrict__ cnt,
                                               const uint2* __restrict__ tset, uint32_t* __restrict__ tcur,
                                               const uint2* __restrict__ ranges, Status* __restrict__ st,
                                               unsigned long long* __restrict__ pkey) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ uint32_t s_pos[kAggTiles];
  if (st->overflow) return;
  const int64_t item = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const AggWin aw = agg_window(*D);
  uint32_t c = 0;
  const FrameDev* F = nullptr;
  unsigned long long k = 0;
  // the item's tiles: its stored set, or (a set that is not one range) the
  // counting pass's enumeration repeated from the geometry
  TileSet ts{0, -1, 0, 0};
  bool slow = false;
  BinGeom g;
  float4 pb = make_float4(0.f, 0.f, 0.f, 0.f);
  if (item < D->n_items) {
    c = cnt[item];
    if (c) {
      const int f = frame_of_item(*D, item);
      F = &D->f[f];
      k = (static_cast<unsigned long long>(key[item]) << 32) | static_cast<uint32_t>(item);
      const uint2 packed = tset[item];
      slow = packed.x == kTsEnumerate;
      if (slow) {
        const MapDev& M = D->m[F->map];
        const int64_t i = item - F->item_base;
        bin_geom(M.mean + 3 * i, M.ls + 2 * i, *F, g);
        pb = pixel_box(g, *F);   // the sphere box the counting pass used (the stored box is the culling box)
      } else {
        ts = unpack_set(packed);
      }
    }
  }
  const auto tiles = [&](auto fn) -> uint32_t {
    if (slow) return for_each_tile(g, *F, tab, pb, fn);
    for_each_in_set(ts, *F, fn);
    return static_cast<uint32_t>((ts.r1 - ts.r0 + 1) * ts.nc);
  };
  // the enumeration repeats the counting pass exactly, so every slot lies
  // inside the tile's run; a slot outside it is dropped and recorded
  const auto put = [&](uint32_t t, uint32_t pos) {
    if (pos < ranges[t].y) pkey[pos] = k;
    else st->check = 1u;
  };
  if (!aw.local) {
    if (c) {
      const uint32_t n = tiles([&](uint32_t t) { put(t, atomicAdd(tcur + t, 1u)); });
      if (n != c) st->check = 1u;
    }
    return;
  }
  // shared counters: count, reserve one run per touched tile (the counter
  // becomes the run's next slot), then fill it
  for (uint32_t t = threadIdx.x; t < aw.n; t += blockDim.x) s_pos[t] = 0u;
  __syncthreads();
  if (c) {
    const uint32_t n = tiles([&](uint32_t t) { atomicAdd(s_pos + (t - aw.base), 1u); });
    if (n != c) st->check = 1u;
  }
  __syncthreads();
  for (uint32_t t = threadIdx.x; t < aw.n; t += blockDim.x) {
    const uint32_t m = s_pos[t];
    if (m) s_pos[t] = atomicAdd(tcur + aw.base + t, m);
  }
  __syncthreads();
  if (c) tiles([&](uint32_t t) { put(t, atomicAdd(s_pos + (t - aw.base), 1u)); });
}

// ---------------------------------------------------------------------------
// Per-tile sort
// ---------------------------------------------------------------------------
// ---- up to 2048 keys in shared memory: distribution sort --------------------
// The depths of a bucket are spread by an estimate of their rank: 256 coarse
// bins linear in the depth bits are counted, and inside its coarse bin a key
// takes the linearly interpolated one of as many fine bins as the bin has
// keys (about one key per fine bin unless the depths cluster far below a
// coarse bin's width).  Both maps are monotone in the depth, so the keys of
// one fine bin are adjacent in the result: they are placed together and each
// finds its rank by comparing the 64-bit keys of its bin.  A bucket with more
// than kDense keys in one fine bin (mostly equal depths) takes a bitonic sort up
// to kBitonicMax keys, a merge sort beyond.  Bound by issue and by its nine
// barriers, at about 60 instructions per key; a merge sort, one pass per
// doubling, took 28 us on the street frame (1.27 M keys in 1,916 buckets) and
// 524 us on 8 keyframes of a 1M map (21.6 M keys in buckets up to 2,048), this 18
// and 113 us.
constexpr int kSortCta = 256;
constexpr int kSortPer = kSortMax / kSortCta;
constexpr uint32_t kCoarse = 256;
constexpr uint32_t kDense = 64;
// (200 tiles of 100 equal depths, the binning: 31.4 us, merged 33.4; of 2,000
// equal depths 75.7 and 61.4)
constexpr uint32_t kBitonicMax = 256;
static_assert(kCoarse == kSortCta && kSortPer == 8, "one coarse bin per thread, eight fine bins per thread");

struct SortSmem {
  unsigned long long key[kSortMax];
  alignas(16) uint32_t fine[kSortMax + 4];
  uint32_t coarse[kCoarse + 1];
  uint32_t red[4][kSortCta / 32];
};

// A depth's coarse bin and its place inside it ([0, 1] up to rounding): the
// depth bits above `lo`, scaled to the number of bins.
struct DepthMap {
  uint32_t lo;
  float scale;
  uint32_t last;   // the last bin
  __device__ __forceinline__ DepthMap(uint32_t lo_, uint32_t hi, uint32_t bins)
      : lo(lo_), scale(static_cast<float>(bins) / (static_cast<float>(hi - lo_) + 1.0f)), last(bins - 1) {}
  __device__ __forceinline__ uint32_t bin(uint32_t d, float& frac) const {
    // (rounded operations: every call gives a depth the same bin)
    const float x = fmul(static_cast<float>(d - lo), scale);
    const uint32_t c = min(static_cast<uint32_t>(x), last);
    frac = fsub(x, static_cast<float>(c));
    return c;
  }
  // Estimated rank from the bins' exclusive counts: monotone in d.
  __device__ __forceinline__ uint32_t rank(uint32_t d, const uint32_t* start) const {
    float frac;
    const uint32_t c = bin(d, frac);
    const uint32_t b = start[c], m = start[c + 1] - b;
    return b + min(static_cast<uint32_t>(fmul(frac, static_cast<float>(m))), m - 1u);
  }
};

// Exclusive prefix of v over the CTA (kSortCta threads); s_w: a word per
// warp.  Holds one barrier.
__device__ __forceinline__ uint32_t cta_exclusive(uint32_t v, uint32_t* s_w) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_w[wid] = incl;
  __syncthreads();
  uint32_t base = incl - v;
#pragma unroll
  for (int w = 0; w < kSortCta / 32; ++w) base += w < wid ? s_w[w] : 0u;
  return base;
}

// Ascending bitonic sort of key[0, n) in shared memory, n <= kSortMax, padded
// with the largest key.  Every thread of the CTA calls it.
__device__ __noinline__ void smem_bitonic(unsigned long long* key, uint32_t n) {
  uint32_t N = 2;
  while (N < n) N <<= 1;
  for (uint32_t i = n + threadIdx.x; i < N; i += kSortCta) key[i] = ~0ull;
  __syncthreads();
  for (uint32_t w = 2; w <= N; w <<= 1)
    for (uint32_t j = w >> 1; j; j >>= 1) {
      for (uint32_t t = threadIdx.x; t < N / 2; t += kSortCta) {
        const uint32_t i = 2 * t - (t & (j - 1)), o = i + j;   // (bit j of i is clear)
        const unsigned long long a = key[i], b = key[o];
        if ((a > b) == ((i & w) == 0)) {
          key[i] = b;
          key[o] = a;
        }
      }
      __syncthreads();
    }
}

__device__ __forceinline__ void cas_reg(unsigned long long& a, unsigned long long& b) {
  const unsigned long long x = a, y = b;
  a = x > y ? y : x;
  b = x > y ? x : y;
}

// Shared-memory index of merged key x: one slot left free after every 8 keys, so
// that the 8-key rows of consecutive threads start in different banks.
__device__ __forceinline__ uint32_t pad8(uint32_t x) { return x + (x >> 3); }
static_assert(sizeof(SortSmem) >= 8 * (kSortMax + kSortMax / 8), "the merge sort's rows reach past the keys");

// Merge sort of s.key[0, n), 0 < n <= kSortMax; key i is left at s.key[pad8(i)]
// (over the bins).  Every thread sorts 8 keys in registers (Batcher's odd-even
// merge network), then pairs of runs are merged, every thread 8 outputs from
// their merge-path start, read into registers before any is stored.  Every
// thread of the CTA calls it after a barrier; it ends with one.
__device__ __noinline__ void smem_merge(SortSmem& s, uint32_t n) {
  const uint32_t t = threadIdx.x, rows = (n + 7) / 8, N = 8 * rows;
  unsigned long long* const buf = s.key;
  unsigned long long k[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) k[r] = t < rows && t + r * rows < n ? buf[t + r * rows] : ~0ull;
  cas_reg(k[0], k[1]); cas_reg(k[2], k[3]); cas_reg(k[4], k[5]); cas_reg(k[6], k[7]);
  cas_reg(k[0], k[2]); cas_reg(k[1], k[3]); cas_reg(k[4], k[6]); cas_reg(k[5], k[7]);
  cas_reg(k[1], k[2]); cas_reg(k[5], k[6]);
  cas_reg(k[0], k[4]); cas_reg(k[1], k[5]); cas_reg(k[2], k[6]); cas_reg(k[3], k[7]);
  cas_reg(k[2], k[4]); cas_reg(k[3], k[5]);
  cas_reg(k[1], k[2]); cas_reg(k[3], k[4]); cas_reg(k[5], k[6]);
  __syncthreads();
  if (t < rows)
#pragma unroll
    for (int r = 0; r < 8; ++r) buf[9 * t + r] = k[r];
  for (uint32_t L = 8; L < N; L <<= 1) {
    // (up to L = 128 the threads of a pair of runs are of one warp)
    if (L <= 128) __syncwarp();
    else __syncthreads();
    if (t < rows) {
      const uint32_t d = 8 * t & (2 * L - 1);   // first output in the pair
      const uint32_t a0 = 8 * t - d, b0 = a0 + L;
      const uint32_t la = min(L, N - a0), lb = b0 < N ? min(L, N - b0) : 0u;
      uint32_t lo = d > lb ? d - lb : 0u, hi = d < la ? d : la;
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (buf[pad8(a0 + mid)] > buf[pad8(b0 + d - mid - 1)]) hi = mid;
        else lo = mid + 1;
      }
      uint32_t i = lo, j = d - lo;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        // (ties, which only the padding has, go to the first run, as in the search)
        const unsigned long long a = i < la ? buf[pad8(a0 + i)] : ~0ull, b = j < lb ? buf[pad8(b0 + j)] : ~0ull;
        const bool first = j >= lb || (i < la && a <= b);
        k[r] = first ? a : b;
        i += first;
        j += !first;
      }
    }
    if (L <= 128) __syncwarp();
    else __syncthreads();
    if (t < rows)
#pragma unroll
      for (int r = 0; r < 8; ++r) buf[9 * t + r] = k[r];
  }
  __syncthreads();
}

// The n <= kSortMax keys get(0) .. get(n - 1) sorted, their items written to
// out (get may read what out overwrites: every key is read first).  Called by
// the whole CTA; the caller separates two calls by a barrier.
template <bool MERGE, class Get>
__device__ __forceinline__ void sort_small(const Get& get, uint32_t n, uint32_t* out, SortSmem& s) {
  const uint32_t t = threadIdx.x;
  const int wid = t >> 5;
  unsigned long long k[kSortPer];
  uint32_t lo = ~0u, hi = 0u;
#pragma unroll
  for (int r = 0; r < kSortPer; ++r) {
    const uint32_t i = r * kSortCta + t;
    if (i < n) {
      k[r] = get(i);
      lo = min(lo, static_cast<uint32_t>(k[r] >> 32));
      hi = max(hi, static_cast<uint32_t>(k[r] >> 32));
    }
  }
  for (uint32_t i = t; i < n; i += kSortCta) s.fine[i] = 0u;
  s.coarse[t] = 0u;
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if ((t & 31) == 0) {
    s.red[0][wid] = lo;
    s.red[1][wid] = hi;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kSortCta / 32; ++w) {
    lo = min(lo, s.red[0][w]);
    hi = max(hi, s.red[1][w]);
  }
  const DepthMap map(lo, hi, kCoarse);
#pragma unroll
  for (int r = 0; r < kSortPer; ++r)
    if (r * kSortCta + t < n) {
      float frac;
      atomicAdd(&s.coarse[map.bin(static_cast<uint32_t>(k[r] >> 32), frac)], 1u);
    }
  __syncthreads();
  const uint32_t base = cta_exclusive(s.coarse[t], s.red[2]);
  s.coarse[t] = base;   // (every thread has read its own count only)
  if (t == 0) s.coarse[kCoarse] = n;
  __syncthreads();
  uint32_t fo[kSortPer];   // fine bin and the key's place among the bin's arrivals
#pragma unroll
  for (int r = 0; r < kSortPer; ++r)
    if (r * kSortCta + t < n) {
      const uint32_t f = map.rank(static_cast<uint32_t>(k[r] >> 32), s.coarse);
      fo[r] = f | (atomicAdd(&s.fine[f], 1u) << 16);
    }
  __syncthreads();
  uint32_t v[8], sum = 0u, most = 0u;
  uint4* f4 = reinterpret_cast<uint4*>(s.fine) + 2 * t;
  if (8 * t < n) {
    const uint4 a = f4[0], b = f4[1];
    const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      v[j] = 8 * t + j < n ? x[j] : 0u;   // (words past n are not set)
      sum += v[j];
      most = max(most, v[j]);
    }
  }
  uint32_t at = cta_exclusive(sum, s.red[3]);
  if (8 * t < n) {
    uint32_t e[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      e[j] = at;
      at += v[j];
    }
    f4[0] = make_uint4(e[0], e[1], e[2], e[3]);
    f4[1] = make_uint4(e[4], e[5], e[6], e[7]);
    if (8 * t + 8 >= n) s.fine[n] = n;
  }
  const bool dense = __syncthreads_or(most > kDense);
#pragma unroll
  for (int r = 0; r < kSortPer; ++r)
    if (r * kSortCta + t < n) s.key[s.fine[fo[r] & 0xffffu] + (fo[r] >> 16)] = k[r];
  __syncthreads();
  if (dense) {
    // (MERGE: in the tiles' kernel; the groups' one would need more registers
    // for it, 5 % of six batched maps' step)
    const bool merge = MERGE && n > kBitonicMax;
    if (merge) smem_merge(s, n);
    else smem_bitonic(s.key, n);
    for (uint32_t i = t; i < n; i += kSortCta) out[i] = static_cast<uint32_t>(s.key[merge ? pad8(i) : i]);
    return;
  }
  for (uint32_t i = t; i < n; i += kSortCta) {
    const unsigned long long x = s.key[i];
    const uint32_t f = map.rank(static_cast<uint32_t>(x >> 32), s.coarse);
    const uint32_t b = s.fine[f], e = s.fine[f + 1];
    uint32_t pos = b;
    if (e - b > 1)
      for (uint32_t j = b; j < e; ++j) pos += s.key[j] < x;
    out[pos] = static_cast<uint32_t>(x);
  }
}

// ---- buckets beyond 2048 keys: partitioned into groups ------------------------
// k_long_split: one CTA takes a bucket (claimed in the tile scan's
// longest-first order).  A depth map like the one above with kLongCoarse bins estimates
// every key's rank, and the keys of one group of 2^sh estimated ranks (1,024,
// more beyond 2 M keys) are scattered to one range of a second key buffer made
// of the pair-tile and item arrays (high and low 32 bits; the pair tiles are
// rewritten on request only).  Then k_tile_sort sorts the groups of all
// buckets, one CTA each, like short buckets.  The split is a few reads of the keys
// by 1,024 threads, short even for the longest bucket, and everything after
// it is spread over the chip; one CTA per bucket, merging chunks through
// global memory, was bound by the longest bucket's serial passes (6 maps with
// buckets up to 292 k keys, 28.9 M long keys: 3.49 -> 0.58 + 0.27 ms; 8
// keyframes of a 1M map, 25.6 M long keys: 1.04 -> 0.18 + 0.25 ms).
// A bucket with a group of more than kSortMax keys is partitioned anew, by the same
// CTA when its other buckets are done: while one bin holds most keys (a smooth wall
// in a bucket with a near and a far surfel) the bins are spread over its range
// alone, and a group that is still too large (several such clusters, or equal
// depths) is partitioned once more with its own range of (depth, item).  What then
// still exceeds kSortMax (clusters within clusters) is sorted by its CTA with sorted
// chunks and merge passes through global memory.  (10,000 keys on a wall with 1 mm
// of noise between a near and a far surfel, the binning: 196 us when the large
// groups were merged, 74 with one CTA per bucket, now 59; 300,000 equal depths 7.8,
// 3.1 and 0.85 ms.  All of it stays out of the loop over the buckets, which has 32
// registers: a call in it made the longest bucket of six maps 499 -> 776 us alone,
// its loads no longer four at a time.)
constexpr int kLongCta = 1024;
constexpr uint32_t kLongCoarse = 2048;
constexpr uint32_t kMaxGroups = 2048;
constexpr uint32_t kGroupBits = 10;
static_assert(kLongCoarse == 2 * kLongCta && kMaxGroups == 2 * kLongCta, "two bins or groups per thread");

// A bucket's keys: 64-bit words, or split into high and low 32-bit halves
// (read from L2: the CTA rewrites them).
struct KeyBuf {
  unsigned long long* k;
  uint32_t *hi, *lo;
  __device__ __forceinline__ unsigned long long get(uint32_t i) const {
    return k ? __ldcg(k + i) : (static_cast<unsigned long long>(__ldcg(hi + i)) << 32) | __ldcg(lo + i);
  }
  __device__ __forceinline__ void put(uint32_t i, unsigned long long v) const {
    if (k) {
      k[i] = v;
    } else {
      hi[i] = static_cast<uint32_t>(v >> 32);
      lo[i] = static_cast<uint32_t>(v);
    }
  }
};

// Merge-path split: how many of the first d outputs of merging A[0, la) and
// B[0, lb) come from A (keys are distinct).
__device__ __forceinline__ uint32_t path_split(const KeyBuf& X, uint32_t a0, uint32_t la, uint32_t b0, uint32_t lb,
                                               uint32_t d) {
  uint32_t lo = d > lb ? d - lb : 0u, hi = d < la ? d : la;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (X.get(a0 + mid) > X.get(b0 + d - mid - 1)) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

// The n keys of Y sorted by one CTA, their items left in Y.lo: chunks of
// kSortMax keys sorted in shared memory into X, then passes that merge pairs
// of runs, ping-ponging between X and Y, in output tiles of kSortMax keys (the
// tiles' first merge-path diagonals found by binary searches, one per thread,
// their two input ranges loaded into shared memory, eight outputs merged per
// thread).
__device__ __noinline__ void merge_sort_global(const KeyBuf& X, const KeyBuf& Y, uint32_t n, SortSmem& s) {
  const uint32_t t = threadIdx.x;
  unsigned long long* sa = s.key;
  uint32_t* s_split = s.fine;   // kSortCta + 1 words
  for (uint32_t c0 = 0; c0 < n; c0 += kSortMax) {
    const uint32_t m = min(kSortMax, n - c0);
    for (uint32_t i = t; i < m; i += kSortCta) sa[i] = Y.get(c0 + i);
    __syncthreads();
    smem_bitonic(sa, m);
    for (uint32_t i = t; i < m; i += kSortCta) X.put(c0 + i, sa[i]);
    __syncthreads();
  }
  bool in_x = true;
  for (uint32_t R = kSortMax; R < n; R <<= 1) {
    const KeyBuf& S = in_x ? X : Y;
    const KeyBuf& Dst = in_x ? Y : X;
    const uint32_t n_out = (n + kSortMax - 1) / kSortMax;   // output tiles (a run pair holds whole tiles)
    for (uint32_t q0 = 0; q0 < n_out; q0 += kSortCta) {
      // first diagonal of output tiles q0 + t (and the end of the last one)
      __syncthreads();
      for (uint32_t q = q0 + t; q <= min(q0 + kSortCta, n_out); q += kSortCta) {
        const uint32_t o = min(q * kSortMax, n);
        uint32_t p = o / (2 * R);
        if (o == n && o % (2 * R) == 0 && o > 0) --p;   // the end diagonal of the last pair
        const uint32_t a0 = 2 * R * p, la = min(R, n - a0), b0 = a0 + R;
        const uint32_t lb = b0 < n ? min(R, n - b0) : 0u;
        s_split[q - q0] = path_split(S, a0, la, b0, lb, o - a0);
      }
      __syncthreads();
      const uint32_t q1 = min(q0 + kSortCta, n_out);
      for (uint32_t q = q0; q < q1; ++q) {
        const uint32_t o = q * kSortMax, oe = min(o + kSortMax, n);
        const uint32_t p = o / (2 * R);
        const uint32_t a0 = 2 * R * p, la = min(R, n - a0), b0 = a0 + R;
        const uint32_t d0 = o - a0, d1 = oe - a0;
        const uint32_t i0 = s_split[q - q0];
        // the tile's end diagonal: the next tile's first one, or the whole
        // pair when the tile closes it
        const uint32_t i1 = d1 == la + (b0 < n ? min(R, n - b0) : 0u) ? la : s_split[q + 1 - q0];
        const uint32_t j0 = d0 - i0, j1 = d1 - i1;
        const uint32_t na = i1 - i0, nb = j1 - j0;
        // A's part then B's part, in shared memory
        for (uint32_t i = t; i < na; i += kSortCta) sa[i] = S.get(a0 + i0 + i);
        for (uint32_t i = t; i < nb; i += kSortCta) sa[na + i] = S.get(b0 + j0 + i);
        __syncthreads();
        const uint32_t d = 8 * t;
        if (d < na + nb) {
          uint32_t lo = d > nb ? d - nb : 0u, hi = d < na ? d : na;
          while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (sa[mid] > sa[na + d - mid - 1]) hi = mid;
            else lo = mid + 1;
          }
          uint32_t i = lo, j = d - lo;
          const uint32_t cnt = min(8u, na + nb - d);
          for (uint32_t r = 0; r < cnt; ++r) {
            const unsigned long long a = i < na ? sa[i] : ~0ull, b = j < nb ? sa[na + j] : ~0ull;
            const bool takeA = j >= nb || (i < na && a < b);
            Dst.put(o + d + r, takeA ? a : b);
            i += takeA;
            j += !takeA;
          }
        }
        __syncthreads();
      }
    }
    in_x = !in_x;
  }
  // the item list: the keys' low halves (already in place when the result is
  // in the split buffer)
  if (in_x)
    for (uint32_t i = t; i < n; i += kSortCta) Y.lo[i] = static_cast<uint32_t>(X.get(i));
}

// What k_long_split writes for the forward's long lists (SegBuf).
struct SegPlan {
  const uint32_t* longt;
  uint32_t* sbase;
  uint2* segs;
  uint32_t* dead;
  uint32_t blocks;   // warp blocks per tile
};

// fn(key) for n keys in turn, four loads in flight per thread.
template <class Fn>
__device__ __forceinline__ void for_keys(const unsigned long long* X, uint32_t n, Fn fn) {
  for (uint32_t i0 = threadIdx.x; i0 < n; i0 += 4 * kLongCta) {
    unsigned long long x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = i0 + u * kLongCta < n ? X[i0 + u * kLongCta] : 0ull;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u * kLongCta < n) fn(x[u]);
  }
}

template <class Fn>
__device__ __forceinline__ void for_keys(const KeyBuf& Y, uint32_t n, Fn fn) {
  for (uint32_t i0 = threadIdx.x; i0 < n; i0 += 2 * kLongCta) {
    const unsigned long long a = Y.get(i0), b = i0 + kLongCta < n ? Y.get(i0 + kLongCta) : 0ull;
    fn(a);
    if (i0 + kLongCta < n) fn(b);
  }
}

// Exclusive prefix over the CTA's 2 * kLongCta words, two per thread (c[2t],
// c[2t + 1]).  Holds two barriers.
__device__ __forceinline__ uint2 long_exclusive(uint2 c, uint32_t* s_w) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t incl = c.x + c.y;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_w[wid] = incl;
  __syncthreads();
  uint32_t w = s_w[lane];
  w = __reduce_add_sync(0xffffffffu, lane < wid ? w : 0u);
  __syncthreads();   // s_w is rewritten by the next call
  const uint32_t b = w + incl - c.x - c.y;
  return make_uint2(b, b + c.x);
}

// The segments of the forward's long lists (one CTA): every list's first
// segment and the (list, segment) items ordered by segment (up to kSegClass;
// the later ones together).
constexpr uint32_t kSegClass = 2 * kLongCta - 1;

__device__ void plan_segments(const uint2* __restrict__ ranges, Status* __restrict__ st, const SegPlan& P,
                              uint32_t* s_cnt, uint32_t* s_w) {
  const uint32_t t = threadIdx.x, n_long = st->n_long;
  const auto segments = [&](uint32_t l) {
    const uint2 rg = ranges[P.longt[l]];
    return (rg.y - rg.x + kSeg - 1) / kSeg;
  };
  s_cnt[2 * t] = s_cnt[2 * t + 1] = 0u;
  __syncthreads();
  uint32_t carry = 0;
  for (uint32_t l0 = 0; l0 < n_long; l0 += kLongCta) {
    const uint32_t l = l0 + t;
    const uint32_t n = l < n_long ? segments(l) : 0u;
    const uint32_t at = long_exclusive(make_uint2(n, 0u), s_w).x;
    if (n) {
      P.sbase[P.longt[l]] = carry + at;
      for (uint32_t s = 0; s < n; ++s) atomicAdd(&s_cnt[min(s, kSegClass)], 1u);
    }
    if (t == kLongCta - 1) s_w[0] = at + n;
    __syncthreads();
    carry += s_w[0];
    __syncthreads();
  }
  const uint2 first = long_exclusive(make_uint2(s_cnt[2 * t], s_cnt[2 * t + 1]), s_w);
  s_cnt[2 * t] = first.x;
  s_cnt[2 * t + 1] = first.y;
  __syncthreads();
  for (uint32_t l = t; l < n_long; l += kLongCta) {
    const uint32_t n = segments(l);
    for (uint32_t s = 0; s < n; ++s) P.segs[atomicAdd(&s_cnt[min(s, kSegClass)], 1u)] = make_uint2(l, s);
  }
  for (uint32_t i = t; i < n_long * P.blocks * 32; i += kLongCta) P.dead[i] = ~0u;
  if (t == 0) st->n_segs = carry;
  __syncthreads();
}

// Bins of the values above `base` (those below count as base, those beyond the
// last bin as its end), monotone in the value: rounded conversion and product.
template <class V>
struct Bins {
  V base;
  float scale;
  __device__ __forceinline__ uint32_t bin(V v, float& frac) const {
    const float x = fmul(static_cast<float>(max(v, base) - base), scale);
    const uint32_t c = min(static_cast<uint32_t>(x), kLongCoarse - 1u);
    frac = fsub(x, static_cast<float>(c));
    return c;
  }
  // Estimated rank from the bins' exclusive counts: monotone in v.
  __device__ __forceinline__ uint32_t rank(V v, const uint32_t* start) const {
    float frac;
    const uint32_t c = bin(v, frac);
    const uint32_t b = start[c], m = start[c + 1] - b;
    return b + min(static_cast<uint32_t>(fmul(frac, static_cast<float>(m))), m - 1u);
  }
  __device__ __forceinline__ bool wide() const { return scale < 0.25f; }   // more than four values a bin
  // All bins over the range of bin c (and a little more: the bounds are rounded).
  __device__ __forceinline__ void narrow(uint32_t c) {
    const float width = 1.0f / scale;
    base += static_cast<V>(fmaxf((static_cast<float>(c) - 0.02f) * width, 0.0f));
    scale = static_cast<float>(kLongCoarse) / (1.04f * width + 1.0f);
  }
};

template <class V>
__device__ __forceinline__ Bins<V> bins_over(V lo, V hi) {
  return Bins<V>{lo, static_cast<float>(kLongCoarse) / (static_cast<float>(hi - lo) + 1.0f)};
}

struct SplitSmem {
  uint32_t hist[2 * kLongCta];       // counts per bin, then per group, then group cursors
  uint32_t start[kLongCoarse + 2];   // the keys before each bin
  uint32_t w[32], mm[4], claim, at, next;
  uint32_t clustered;   // head of the list of this CTA's clustered buckets (1 + order position, 0 at the end)
};

// One partition of n keys: each(fn) calls fn(value, key) for all of them, the
// bins estimate ranks, and the keys of one group of 2^sh estimated ranks go to
// one range: put(place, key).  While one bin holds most keys, the bins are
// spread over its range alone.  early(counts, first places) gets the thread's
// groups 2t and 2t + 1 before the keys move.  hist is zero on entry.
template <class V, class Each, class Early, class Put>
__device__ __forceinline__ void partition(const Each& each, Bins<V> bins, uint32_t n, uint32_t sh, SplitSmem& s,
                                          const Early& early, const Put& put) {
  const uint32_t t = threadIdx.x;
  uint2 c;
  while (true) {
    each([&](V v, unsigned long long) {
      float frac;
      atomicAdd(&s.hist[bins.bin(v, frac)], 1u);
    });
    __syncthreads();
    c = make_uint2(s.hist[2 * t], s.hist[2 * t + 1]);
    // (every round narrows the range by more than a thousand times)
    if (!__syncthreads_or(max(c.x, c.y) > n / 2) || !bins.wide()) break;
    if (max(c.x, c.y) > n / 2) s.next = 2 * t + (c.y > c.x);
    s.hist[2 * t] = s.hist[2 * t + 1] = 0u;
    __syncthreads();
    bins.narrow(s.next);
  }
  const uint2 first = long_exclusive(c, s.w);
  s.start[2 * t] = first.x;
  s.start[2 * t + 1] = first.y;
  if (t == 0) s.start[kLongCoarse] = n;
  s.hist[2 * t] = s.hist[2 * t + 1] = 0u;   // (every thread has read its own counts only)
  __syncthreads();
  each([&](V v, unsigned long long) { atomicAdd(&s.hist[bins.rank(v, s.start) >> sh], 1u); });
  __syncthreads();
  c = make_uint2(s.hist[2 * t], s.hist[2 * t + 1]);
  const uint2 at = long_exclusive(c, s.w);
  s.hist[2 * t] = at.x;
  s.hist[2 * t + 1] = at.y;
  early(c, at);
  __syncthreads();
  each([&](V v, unsigned long long x) { put(atomicAdd(&s.hist[bins.rank(v, s.start) >> sh], 1u), x); });
}

__device__ __forceinline__ uint32_t group_shift(uint32_t n) {
  uint32_t sh = kGroupBits;
  while (((n - 1) >> sh) >= kMaxGroups) ++sh;
  return sh;
}

// The second partition, of the n keys at `first` of the split buffer (the arrays'
// pointers are those of this range; through the key array, which the first one is
// done with): by (depth, item) as one number, the depths above the lowest times the
// items' span plus the item, so that equal depths spread by item.
__device__ __noinline__ void split_again(SplitSmem& s, uint32_t first, uint32_t n, unsigned long long* pkey,
                                         uint32_t* ptile, uint32_t* pv, uint2* groups, uint32_t* all_groups) {
  const uint32_t t = threadIdx.x;
  const KeyBuf Y{nullptr, ptile, pv};
  if (t < 4) s.mm[t] = t & 1u ? 0u : ~0u;
  s.hist[2 * t] = s.hist[2 * t + 1] = 0u;
  __syncthreads();
  uint32_t dlo = ~0u, dhi = 0u, ilo = ~0u, ihi = 0u;
  for_keys(Y, n, [&](unsigned long long x) {
    dlo = min(dlo, static_cast<uint32_t>(x >> 32));
    dhi = max(dhi, static_cast<uint32_t>(x >> 32));
    ilo = min(ilo, static_cast<uint32_t>(x));
    ihi = max(ihi, static_cast<uint32_t>(x));
  });
  dlo = __reduce_min_sync(0xffffffffu, dlo);
  dhi = __reduce_max_sync(0xffffffffu, dhi);
  ilo = __reduce_min_sync(0xffffffffu, ilo);
  ihi = __reduce_max_sync(0xffffffffu, ihi);
  if ((t & 31) == 0) {
    atomicMin(&s.mm[0], dlo);
    atomicMax(&s.mm[1], dhi);
    atomicMin(&s.mm[2], ilo);
    atomicMax(&s.mm[3], ihi);
  }
  __syncthreads();
  dlo = s.mm[0];
  ilo = s.mm[2];
  const unsigned long long span = static_cast<unsigned long long>(s.mm[3] - ilo) + 1ull;
  const unsigned long long most = (s.mm[1] - dlo) * span + (span - 1ull);
  const uint32_t sh = group_shift(n), n_groups = ((n - 1) >> sh) + 1;
  if (t == 0) s.at = atomicAdd(all_groups, n_groups);
  partition([&](auto fn) {
              for_keys(Y, n, [&](unsigned long long x) {
                fn((static_cast<uint32_t>(x >> 32) - dlo) * span + (static_cast<uint32_t>(x) - ilo), x);
              });
            },
            bins_over(0ull, most), n, sh, s,
            [&](uint2 c, uint2 at) {
              if (2 * t < n_groups) groups[s.at + 2 * t] = make_uint2(first + at.x, first + at.x + c.x);
              if (2 * t + 1 < n_groups) groups[s.at + 2 * t + 1] = make_uint2(first + at.y, first + at.y + c.y);
            },
            [&](uint32_t pos, unsigned long long x) { pkey[pos] = x; });
  __syncthreads();
  for (uint32_t i = t; i < n; i += kLongCta) Y.put(i, __ldcg(pkey + i));
}

// The first bucket of the CTA's list, whose depths cluster: partitioned with bins
// spread over the cluster, then the groups of more than kSortMax keys once more,
// one after the other.
__device__ __noinline__ void split_clustered(SplitSmem& s, unsigned long long* pkey, uint32_t* ptile, uint32_t* pv,
                                             uint2* groups, uint32_t* all_groups, const uint2* ranges,
                                             const uint32_t* order, const uint32_t* next) {
  const uint32_t t = threadIdx.x, k = s.clustered - 1;
  const uint2 rg = ranges[order[k]];
  const uint32_t first = rg.x, n = rg.y - rg.x;
  const uint32_t sh = group_shift(n), n_groups = ((n - 1) >> sh) + 1;
  const unsigned long long* X = pkey + first;
  __syncthreads();   // (every thread has read the list's head)
  if (t == 0) {
    s.clustered = next[k];
    s.mm[0] = ~0u;
    s.mm[1] = 0u;
  }
  __syncthreads();
  uint32_t lo = ~0u, hi = 0u;
  for_keys(X, n, [&](unsigned long long x) {
    lo = min(lo, static_cast<uint32_t>(x >> 32));
    hi = max(hi, static_cast<uint32_t>(x >> 32));
  });
  atomicMin(&s.mm[0], __reduce_min_sync(0xffffffffu, lo));
  atomicMax(&s.mm[1], __reduce_max_sync(0xffffffffu, hi));
  if (t == 0) s.at = atomicAdd(all_groups, n_groups);
  s.hist[2 * t] = s.hist[2 * t + 1] = 0u;
  __syncthreads();
  partition([&](auto fn) { for_keys(X, n, [&](unsigned long long x) { fn(static_cast<uint32_t>(x >> 32), x); }); },
            bins_over(s.mm[0], s.mm[1]), n, sh, s,
            [&](uint2 c, uint2 at) {
              // (an empty range where split_again stores the groups instead)
              const uint2 e = make_uint2(c.x > kSortMax ? 0u : c.x, c.y > kSortMax ? 0u : c.y);
              if (2 * t < n_groups) groups[s.at + 2 * t] = make_uint2(first + at.x, first + at.x + e.x);
              if (2 * t + 1 < n_groups) groups[s.at + 2 * t + 1] = make_uint2(first + at.y, first + at.y + e.y);
            },
            [&](uint32_t pos, unsigned long long x) {
              ptile[first + pos] = static_cast<uint32_t>(x >> 32);
              pv[first + pos] = static_cast<uint32_t>(x);
            });
  __syncthreads();
  // (every cursor stands at its group's end, where the next group starts)
  const uint32_t a = t ? s.hist[2 * t - 1] : 0u;
  const uint2 end = make_uint2(s.hist[2 * t], s.hist[2 * t + 1]), c = make_uint2(end.x - a, end.y - end.x);
  for (uint32_t from = 0;;) {
    __syncthreads();
    if (t == 0) s.next = ~0u;
    __syncthreads();
    if (c.y > kSortMax && 2 * t + 1 >= from) atomicMin(&s.next, 2 * t + 1);
    if (c.x > kSortMax && 2 * t >= from) atomicMin(&s.next, 2 * t);
    __syncthreads();
    const uint32_t g = s.next;
    if (g == ~0u) return;   // (after a barrier: the next call may rewrite everything)
    if (t == g / 2) {
      s.mm[0] = g & 1u ? c.y : c.x;
      s.mm[1] = g & 1u ? end.y : end.x;
    }
    __syncthreads();
    const uint32_t m = s.mm[0], e = s.mm[1];
    __syncthreads();
    const uint32_t at = first + e - m;
    split_again(s, at, m, pkey + at, ptile + at, pv + at, groups, all_groups);
    from = g + 1;
  }
}

__global__ void __launch_bounds__(kLongCta, 2)
    k_long_split(const uint2* __restrict__ ranges, Status* __restrict__ st, const uint32_t* __restrict__ order,
                 uint32_t n_tiles, unsigned long long* pkey, uint32_t* __restrict__ ptile,
                 uint32_t* __restrict__ pv, uint2* __restrict__ groups, uint32_t* __restrict__ next, SegPlan plan) {
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ SplitSmem s;
  if (st->overflow || st->n_big == 0) return;
  const uint32_t t = threadIdx.x;
  if (t == 0) s.clustered = 0u;
  if (blockIdx.x == gridDim.x - 1 && st->n_long) plan_segments(ranges, st, plan, s.hist, s.w);
  while (true) {
    // buckets in the tile scan's longest-first order; the long ones come
    // first, so the first list of a shorter class ends the work
    __syncthreads();
    if (t == 0) {
      s.claim = atomicAdd(&st->long_sort_counter, 1u);
      s.mm[0] = ~0u;
      s.mm[1] = 0u;
    }
    s.hist[2 * t] = s.hist[2 * t + 1] = 0u;
    __syncthreads();
    const uint32_t k = s.claim;
    if (k >= n_tiles) break;
    const uint2 rg = ranges[order[k]];
    const uint32_t n = rg.y - rg.x;
    if (order_bucket(n) > order_bucket(kSortMax + 1)) break;   // a shorter class: no long list follows
    if (n <= kSortMax) continue;
    const uint32_t sh = group_shift(n), n_groups = ((n - 1) >> sh) + 1;
    const unsigned long long* X = pkey + rg.x;
    // the bucket's depth range
    uint32_t lo = ~0u, hi = 0u;
    for_keys(X, n, [&](unsigned long long x) {
      lo = min(lo, static_cast<uint32_t>(x >> 32));
      hi = max(hi, static_cast<uint32_t>(x >> 32));
    });
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((t & 31) == 0) {
      atomicMin(&s.mm[0], lo);
      atomicMax(&s.mm[1], hi);
    }
    __syncthreads();
    const DepthMap map(s.mm[0], s.mm[1], kLongCoarse);
    for_keys(X, n, [&](unsigned long long x) {
      float frac;
      atomicAdd(&s.hist[map.bin(static_cast<uint32_t>(x >> 32), frac)], 1u);
    });
    __syncthreads();
    const uint2 first = long_exclusive(make_uint2(s.hist[2 * t], s.hist[2 * t + 1]), s.w);
    s.start[2 * t] = first.x;
    s.start[2 * t + 1] = first.y;
    if (t == 0) s.start[kLongCoarse] = n;
    s.hist[2 * t] = s.hist[2 * t + 1] = 0u;   // (every thread has read its own counts only)
    __syncthreads();
    for_keys(X, n, [&](unsigned long long x) {
      atomicAdd(&s.hist[map.rank(static_cast<uint32_t>(x >> 32), s.start) >> sh], 1u);
    });
    __syncthreads();
    const uint2 c = make_uint2(s.hist[2 * t], s.hist[2 * t + 1]);
    if (__syncthreads_or(max(c.x, c.y) > kSortMax)) {
      // (listed, and partitioned when this CTA's other buckets are done: a call
      // here would cost the loop its registers)
      if (t == 0) {
        next[k] = s.clustered;
        s.clustered = k + 1;
      }
      continue;
    }
    const uint2 at = long_exclusive(c, s.w);
    s.hist[2 * t] = at.x;
    s.hist[2 * t + 1] = at.y;
    if (t == 0) s.at = atomicAdd(&st->n_groups, n_groups);
    __syncthreads();
    if (2 * t < n_groups) groups[s.at + 2 * t] = make_uint2(rg.x + at.x, rg.x + at.x + c.x);
    if (2 * t + 1 < n_groups) groups[s.at + 2 * t + 1] = make_uint2(rg.x + at.y, rg.x + at.y + c.y);
    for_keys(X, n, [&](unsigned long long x) {
      const uint32_t pos = rg.x + atomicAdd(&s.hist[map.rank(static_cast<uint32_t>(x >> 32), s.start) >> sh], 1u);
      ptile[pos] = static_cast<uint32_t>(x >> 32);
      pv[pos] = static_cast<uint32_t>(x);
    });
  }
  while (s.clustered) split_clustered(s, pkey, ptile, pv, groups, &st->n_groups, ranges, order, next);
}

// A bucket of n <= kWarpSort keys sorted by one warp, kWarpKeys keys a lane: a
// key's place is the number of smaller ones.
constexpr int kWarpKeys = kWarpSort / 32;
__device__ __forceinline__ void sort_warp(const unsigned long long* key, uint32_t n, uint32_t* out) {
  const uint32_t lane = threadIdx.x & 31;
  unsigned long long k[kWarpKeys];
  uint32_t rank[kWarpKeys];
#pragma unroll
  for (int q = 0; q < kWarpKeys; ++q) {
    k[q] = lane + 32 * q < n ? key[lane + 32 * q] : ~0ull;
    rank[q] = 0;
  }
#pragma unroll
  for (int p = 0; p < kWarpKeys; ++p)
    for (uint32_t j = 0; j < 32 && j + 32 * p < n; ++j) {
      const unsigned long long x = __shfl_sync(0xffffffffu, k[p], j);
#pragma unroll
      for (int q = 0; q < kWarpKeys; ++q) rank[q] += x < k[q];
    }
#pragma unroll
  for (int q = 0; q < kWarpKeys; ++q)
    if (lane + 32 * q < n) out[rank[q]] = static_cast<uint32_t>(k[q]);
}

// TILES: CTAs below n_tiles take the bucket of their tile, if it has at most
// kSortMax keys.  In a sparse call (below kSparse items a tile) they leave buckets
// of up to kWarpSort keys to a warp each of n_warp more CTAs: with a CTA for every
// tile, a frame of few surfels was bound by 2,048 CTAs' barriers over a few keys
// each.  Binning of a 128 x 1024 frame, without and with the warps: 3,000 surfels 41
// and 35 us, 16,000 42 and 40, 64,000 (31 items a tile) 43.8 and 44.1, 200,000 55.9
// and 57.5; warps up to 128 keys were 2 us slower from 16,000 surfels on.  GROUPS:
// the CTAs after them take the long buckets' groups (their keys in the split
// buffer) in turn.  Both in one kernel take 106 registers, the tiles alone 60, so
// that one is held at 64 (16,000 surfels 49 us with 106, now 40).
constexpr uint32_t kSortWarps = kSortCta / 32;
constexpr int64_t kSparse = 32;
template <bool TILES, bool GROUPS>
__global__ void __launch_bounds__(kSortCta, TILES && GROUPS ? 4 : 0) k_tile_sort(const uint2* __restrict__ ranges,
                                                         const Status* __restrict__ st, uint32_t n_tiles,
                                                         uint32_t n_warp, unsigned long long* pkey, uint32_t* ptile,
                                                         uint32_t* pv, const uint2* __restrict__ groups) {
  if (GROUPS) pdl_wait();   // (launched after k_long_split: wait for it)
  __shared__ SortSmem s;
  if (st->overflow) return;
  const uint32_t tile_ctas = TILES ? n_tiles + n_warp : 0u;
  if (TILES && (!GROUPS || blockIdx.x < tile_ctas)) {
    const bool own = blockIdx.x < n_tiles;
    const uint32_t tile = own ? blockIdx.x : (blockIdx.x - n_tiles) * kSortWarps + (threadIdx.x >> 5);
    if (tile >= n_tiles) return;
    const uint2 rg = ranges[tile];
    const uint32_t n = rg.y - rg.x;
    if (!own) {
      if (n <= kWarpSort) sort_warp(pkey + rg.x, n, pv + rg.x);
    } else if (n > (n_warp ? kWarpSort : 0u) && n <= kSortMax) {   // (longer: k_long_split's)
      sort_small<true>([&](uint32_t i) { return pkey[rg.x + i]; }, n, pv + rg.x, s);
    }
    return;
  }
  if (!GROUPS) return;
  const uint32_t n_groups = st->n_groups;
  for (uint32_t g = blockIdx.x - tile_ctas; g < n_groups; g += gridDim.x - tile_ctas) {
    const uint2 rg = groups[g];
    const uint32_t n = rg.y - rg.x;
    const KeyBuf Y{nullptr, ptile + rg.x, pv + rg.x};
    __syncthreads();   // the previous group's shared memory is no longer read
    if (n == 0) continue;
    if (n <= kSortMax) sort_small<false>([&](uint32_t i) { return Y.get(i); }, n, Y.lo, s);
    else merge_sort_global(KeyBuf{pkey + rg.x, nullptr, nullptr}, Y, n, s);
  }
}

// The tile of every pair (sorted order), written only when a caller asks for
// it (the session's bin read-back): one CTA per tile fills its run.
__global__ void k_fill_tile_of_pair(const uint2* __restrict__ ranges, const Status* __restrict__ st,
                                    uint32_t* __restrict__ ptile) {
  if (st->overflow) return;
  const uint2 rg = ranges[blockIdx.x];
  for (uint32_t i = rg.x + threadIdx.x; i < rg.y; i += blockDim.x) ptile[i] = blockIdx.x;
}

cudaError_t launch_fill_tile_of_pair(const WsPtrs& w, uint32_t n_tiles, cudaStream_t s) {
  if (n_tiles) k_fill_tile_of_pair<<<n_tiles, 256, 0, s>>>(w.ranges, w.st, w.ptile);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Orchestration
// ---------------------------------------------------------------------------
// How the long buckets (more than kSortMax keys) are sorted, by the largest
// map of the call.  None can arise up to kSortMax surfels.  From kSideItems
// surfels on, k_long_split and the groups' sort run on the side stream alongside
// the short buckets' sort; below, inline, without the fork and join that the host
// has to issue.  Binning, inline and side: 3,000 surfels on a 64 x 1024 frame
// 30.9 and 34.6 us, 8,000 32.6 and 34.8, 32,000 34.3 and 35.3, 64,000 36.5 and
// 36.4; on a 128 x 1024 frame 35.0 / 36.3, 37.0 / 37.2, 43.4 / 43.1, 44.3 / 45.0;
// four such frames of 125,000 surfels 322 and 318; 1M surfels, 8 keyframes 0.43 ms
// of long buckets beside 0.11.
constexpr int64_t kSideItems = 32768;
enum LongPath { kLongNone, kLongInline, kLongSide };
static LongPath long_path(int64_t max_n) {
  return max_n <= static_cast<int64_t>(kSortMax) ? kLongNone : (max_n < kSideItems ? kLongInline : kLongSide);
}

// kernels launch_bin enqueues (memsets not counted); max_n: surfels of the
// largest map that a frame renders
int bin_kernel_count(uint32_t n_tiles, int64_t max_n) {
  if (n_tiles == 0) return 4;
  const LongPath p = long_path(max_n);
  return p == kLongNone ? 5 : (p == kLongInline ? 6 : 7);
}

cudaError_t launch_bin(const Layout& L, const WsPtrs& w, int n_frames, int64_t n_items, int64_t max_n,
                       uint32_t n_tiles, uint32_t blocks, const SideStream& side, cudaStream_t s) {
  k_tables<<<n_frames, 256, 0, s>>>(w.desc, w.tables, w.st, reinterpret_cast<uint32_t*>(w.loss_part),
                                    static_cast<uint32_t>(loss_part_bytes() / 4), w.tcur, n_tiles);
  const int64_t ni = n_items > 0 ? n_items : 1;
  const unsigned gi = static_cast<unsigned>((ni + 255) / 256);
  // each of the next three follows a kernel of this chain: dispatched while
  // its predecessor runs, it waits for it in its first instruction
  cudaError_t e0 = launch_dep(k_preprocess, dim3(gi), dim3(256), 0, s, w.desc, w.tables, w.rec, w.box, w.key, w.cnt,
                              w.tset, w.tcur, w.st);
  if (e0 == cudaSuccess)
    e0 = launch_dep(k_tile_scan, dim3(1), dim3(kScanCta), 0, s, w.tcur, n_tiles, w.ranges, w.st, L.pairs_cap, w.work,
                    w.longt, w.cbase);
  if (e0 == cudaSuccess)
    e0 = launch_dep(k_emit, dim3(gi), dim3(256), 0, s, w.desc, w.tables, w.key, w.cnt, w.tset, w.tcur, w.ranges, w.st,
                    w.pkey);
  if (e0 != cudaSuccess) return e0;
  if (n_tiles > 0) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // the short buckets, and the long ones: longest first (an early exit when
    // the tile scan found none), then the CTAs that sort their groups
    const LongPath path = long_path(max_n);
    const unsigned group_ctas = 4 * sms;
    const uint32_t n_warp = n_items < kSparse * n_tiles ? (n_tiles + kSortWarps - 1) / kSortWarps : 0u;
    const SegPlan plan{w.longt, w.sbase, w.segs, w.dead, blocks};
    cudaError_t e = cudaSuccess;
    if (path == kLongInline) {
      k_long_split<<<2 * sms, kLongCta, 0, s>>>(w.ranges, w.st, w.work, n_tiles, w.pkey, w.ptile, w.pv, w.groups,
                                                  w.tcur, plan);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      return launch_dep(k_tile_sort<true, true>, dim3(n_tiles + n_warp + group_ctas), dim3(kSortCta), 0, s, w.ranges, w.st,
                        n_tiles, n_warp, w.pkey, w.ptile, w.pv, w.groups);
    }
    if (path == kLongSide && (e = cudaEventRecord(side.fork, s)) != cudaSuccess) return e;
    k_tile_sort<true, false><<<n_tiles + n_warp, kSortCta, 0, s>>>(w.ranges, w.st, n_tiles, n_warp, w.pkey, w.ptile,
                                                                   w.pv, w.groups);
    if ((e = cudaGetLastError()) != cudaSuccess || path == kLongNone) return e;
    // (the side stream has the higher priority: its CTAs take the slots that
    // short buckets free, and the launches do not delay the short buckets)
    if ((e = cudaStreamWaitEvent(side.s, side.fork, 0)) != cudaSuccess) return e;
    k_long_split<<<2 * sms, kLongCta, 0, side.s>>>(w.ranges, w.st, w.work, n_tiles, w.pkey, w.ptile, w.pv, w.groups,
                                                   w.tcur, plan);
    if ((e = cudaGetLastError()) == cudaSuccess)
      e = launch_dep(k_tile_sort<false, true>, dim3(group_ctas), dim3(kSortCta), 0, side.s, w.ranges, w.st, 0u, 0u,
                     w.pkey, w.ptile, w.pv, w.groups);
    if (e == cudaSuccess) e = cudaEventRecord(side.join, side.s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, side.join, 0);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace lgs
