// lgs_init.cu -- keyframe initialisation of new surfels from a scan (paper
// Sec. 3.2 "Covariance construction and reuse": the k-NN covariance of each
// point and its eigendecomposition; Sec. 3.3: the range-adaptive scale
// initialisation, the physics-based confidence u of Eq. physconf and the
// opacity of Eq. alpha_init).
//
// Launches: the points go into spatial order first (a radix sort by a 27-bit
// Morton code of a uniform grid whose cell is as fine as 27 bits allow for
// the scan's extent), so that a leaf of 32 consecutive points is compact; two
// levels of bounding boxes over them (leaves, nodes of 32 leaves); the k
// nearest neighbours (one warp per query: each lane holds one entry of the
// sorted top 32, boxes and points are tested 32 at a time, nearest box first,
// until no box can hold a closer point); the frame of each point (covariance
// of the neighbourhood, cyclic Jacobi eigendecomposition, scales, confidence,
// opacity, orientation).  Keys carry the original index, so the order of the
// sort never shows in a result.
//
// The neighbour sets are integer outcomes: the squared distance that decides
// them is binary32 ((dx dx + dy dy) + dz dz), each operation correctly
// rounded, ties to the lower index, so the sets are a fixed function of the
// input (and bit-exact against the oracle).  Box pruning is conservative
// (a margin of 1e-5 on the box distance, far above the few ulps that separate
// the box bound from any binary32 distance), so it never changes a set.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "lgs_internal.cuh"

namespace lgs {
namespace {

constexpr uint32_t kIniMaxPoints = 1u << 20;
constexpr int kIniCodeBits = 27;     // Morton code: three radix passes of 9 bits
constexpr int kIniDigit = 9;
constexpr uint32_t kIniBins = 1u << kIniDigit;
constexpr int kIniSortCta = 512;     // one thread per bin
constexpr int kIniSortWarps = kIniSortCta / 32;
constexpr int kIniExtCtas = 128;     // partial extents

struct IniBox {
  float lo[3], hi[3];
};

struct IniParams {
  float R[9], t[3];                  // pose: sensor -> world
  float kappa, s_min, s_max, r0, c0, eps, alpha_min, alpha_max;
  int k;
};

__device__ __forceinline__ void warp_min_max(float (&lo)[3], float (&hi)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
    for (int o = 16; o; o >>= 1) {
      lo[a] = fminf(lo[a], __shfl_xor_sync(0xffffffffu, lo[a], o));
      hi[a] = fmaxf(hi[a], __shfl_xor_sync(0xffffffffu, hi[a], o));
    }
}

// Extent of each CTA's share of the points.
__global__ void __launch_bounds__(256) k_ini_part(const float* __restrict__ pts, uint32_t n, IniBox* __restrict__ part) {
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ float s_lo[8][3], s_hi[8][3];
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float v = pts[3 * i + a];
      lo[a] = fminf(lo[a], v);
      hi[a] = fmaxf(hi[a], v);
    }
  warp_min_max(lo, hi);
  if ((threadIdx.x & 31) == 0)
    for (int a = 0; a < 3; ++a) {
      s_lo[threadIdx.x >> 5][a] = lo[a];
      s_hi[threadIdx.x >> 5][a] = hi[a];
    }
  __syncthreads();
  if (threadIdx.x < 3) {
    float l = INFINITY, h = -INFINITY;
    for (int w = 0; w < 8; ++w) {
      l = fminf(l, s_lo[w][threadIdx.x]);
      h = fmaxf(h, s_hi[w][threadIdx.x]);
    }
    part[blockIdx.x].lo[threadIdx.x] = l;
    part[blockIdx.x].hi[threadIdx.x] = h;
  }
}

// The grid of the Morton code: origin, cell edge and the bits of each axis
// (as many as its extent needs), together at most kIniCodeBits.
struct IniGrid {
  float lo[3], inv_h;
  int bits[3];
  uint32_t top[3];   // largest cell index of each axis
};

__global__ void __launch_bounds__(32) k_ini_grid(const IniBox* __restrict__ part, uint32_t n_part,
                                                 IniGrid* __restrict__ grid) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (uint32_t t = threadIdx.x; t < n_part; t += 32)
    for (int a = 0; a < 3; ++a) {
      lo[a] = fminf(lo[a], part[t].lo[a]);
      hi[a] = fmaxf(hi[a], part[t].hi[a]);
    }
  warp_min_max(lo, hi);
  if (threadIdx.x != 0) return;
  float span[3], most = 1e-20f;
  for (int a = 0; a < 3; ++a) {
    // (an extent beyond binary32 is cut: the code only orders the points)
    span[a] = fminf(hi[a] - lo[a], 1e37f);
    most = fmaxf(most, span[a]);
  }
  // the finest cell most / 2^b whose axes fit: an axis of extent s has
  // floor(s / h) + 1 cells
  IniGrid g;
  for (int b = 21; b >= 1; --b) {
    const float inv_h = static_cast<float>(1 << b) / most * 0.9999f;
    int total = 0;
    for (int a = 0; a < 3; ++a) {
      const float cells = span[a] * inv_h;
      g.top[a] = static_cast<uint32_t>(fminf(cells, static_cast<float>((1 << b) - 1)));
      g.bits[a] = 32 - __clz(g.top[a]);
      g.lo[a] = lo[a];
      total += g.bits[a];
    }
    g.inv_h = inv_h;
    if (total <= kIniCodeBits) break;
  }
  *grid = g;
}

// Morton code over the bits that each axis has, interleaved from the lowest
// bit up (an axis whose bits are used up drops out).
__device__ __forceinline__ uint32_t morton(const uint32_t (&c)[3], const int (&bits)[3]) {
  uint32_t code = 0;
  int at = 0;
  const int most = max(bits[0], max(bits[1], bits[2]));
  for (int b = 0; b < most; ++b)
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (b < bits[a]) code |= ((c[a] >> b) & 1u) << at++;
  return code;
}

// A CTA's share of the sort: R rounds of 512 keys, a contiguous piece of
// 32 R keys per warp (the order within a warp's piece is round, lane).  R = 4
// up to 2^18 points (51 CTAs for a 128 x 1024 scan), 16 beyond, so at most 128
// CTAs: every scatter CTA reads the whole table of counts.
__device__ __forceinline__ uint32_t sort_slot(int R, int r) {
  return blockIdx.x * (kIniSortCta * R) + (threadIdx.x >> 5) * (32 * R) + r * 32 + (threadIdx.x & 31);
}

// Digit counts of a radix pass per CTA: hist[CTA][bin].  The first pass
// (FIRST) also forms the codes.
template <int R, bool FIRST>
__global__ void __launch_bounds__(kIniSortCta) k_ini_count(const float* __restrict__ pts,
                                                           const IniGrid* __restrict__ grid,
                                                           uint32_t* __restrict__ code, const uint2* __restrict__ in,
                                                           uint32_t n, int shift, uint32_t* __restrict__ hist) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ uint32_t s_h[kIniBins];
  s_h[threadIdx.x] = 0;
  __syncthreads();
  IniGrid g;
  if (FIRST) g = *grid;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const uint32_t i = sort_slot(R, r);
    if (i < n) {
      uint32_t k;
      if (FIRST) {
        uint32_t c[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
          c[a] = min(static_cast<uint32_t>(fmaxf((pts[3 * i + a] - g.lo[a]) * g.inv_h, 0.f)), g.top[a]);
        k = morton(c, g.bits);
        code[i] = k;
      } else {
        k = in[i].x;
      }
      atomicAdd(&s_h[(k >> shift) & (kIniBins - 1)], 1u);
    }
  }
  __syncthreads();
  hist[blockIdx.x * kIniBins + threadIdx.x] = s_h[threadIdx.x];
}

// Stable scatter of a radix pass: (code, index) pairs to their places; the
// last pass (LAST) writes the points themselves with their index.  A key's
// place: keys of smaller digits, keys of its digit in earlier CTAs and
// warps, and its rank in its warp's piece.
template <int R, bool FIRST, bool LAST>
__global__ void __launch_bounds__(kIniSortCta) k_ini_scatter(const uint32_t* __restrict__ code,
                                                             const uint2* __restrict__ in, uint32_t n, int shift,
                                                             const uint32_t* __restrict__ hist,
                                                             uint2* __restrict__ out, const float* __restrict__ pts,
                                                             float4* __restrict__ sp) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ uint32_t s_at[kIniSortWarps][kIniBins];
  __shared__ uint32_t s_warp[kIniSortWarps];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int w = 0; w < kIniSortWarps; ++w) s_at[w][threadIdx.x] = 0;
  __syncthreads();
  uint2 kv[R];
  uint32_t rank[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const uint32_t i = sort_slot(R, r);
    kv[r] = i < n ? (FIRST ? make_uint2(code[i], i) : in[i]) : make_uint2(0u, 0u);
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const bool ok = sort_slot(R, r) < n;
    const uint32_t d = ok ? (kv[r].x >> shift) & (kIniBins - 1) : kIniBins;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    uint32_t before = 0;
    if (ok) before = s_at[wid][d];
    __syncwarp();
    if (ok && lane == __ffs(peers) - 1) s_at[wid][d] = before + __popc(peers);
    __syncwarp();
    rank[r] = before + __popc(peers & ((1u << lane) - 1u));
  }
  // thread = bin: its keys in earlier CTAs and in all CTAs
  uint32_t total = 0, mine = 0;
  for (uint32_t b = 0; b < gridDim.x; b += 8) {
    uint32_t v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = b + u < gridDim.x ? hist[(b + u) * kIniBins + threadIdx.x] : 0u;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      total += v[u];
      mine += b + u < blockIdx.x ? v[u] : 0u;
    }
  }
  uint32_t incl = total;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  uint32_t at = mine + incl - total;
  for (int w = 0; w < wid; ++w) at += s_warp[w];
#pragma unroll
  for (int w = 0; w < kIniSortWarps; ++w) {
    const uint32_t c = s_at[w][threadIdx.x];
    s_at[w][threadIdx.x] = at;
    at += c;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (sort_slot(R, r) < n) {
      const uint32_t pos = s_at[wid][(kv[r].x >> shift) & (kIniBins - 1)] + rank[r];
      if (LAST) {
        const uint32_t i = kv[r].y;
        sp[pos] = make_float4(pts[3 * i], pts[3 * i + 1], pts[3 * i + 2], __uint_as_float(i));
      } else {
        out[pos] = kv[r];
      }
    }
  }
}

// Boxes of the leaves (32 points, one warp) and of the nodes (32 leaves, one
// CTA): lo / hi corners as float4, the smallest original index of the points in
// lo.w (as bits).
__global__ void __launch_bounds__(1024) k_ini_boxes(const float4* __restrict__ sp, uint32_t n,
                                                    float4* __restrict__ leaf, float4* __restrict__ node) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ float s_lo[32][3], s_hi[32][3];
  __shared__ uint32_t s_id[32];
  const uint32_t i = blockIdx.x * 1024 + threadIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  uint32_t id = 0xffffffffu;
  if (i < n) {
    const float4 p = sp[i];
    lo[0] = hi[0] = p.x;
    lo[1] = hi[1] = p.y;
    lo[2] = hi[2] = p.z;
    id = __float_as_uint(p.w);
  }
  warp_min_max(lo, hi);
  id = __reduce_min_sync(0xffffffffu, id);
  if (lane == 0) {
    for (int a = 0; a < 3; ++a) {
      s_lo[wid][a] = lo[a];
      s_hi[wid][a] = hi[a];
    }
    s_id[wid] = id;
    if (i < n) {
      leaf[2 * (i >> 5)] = make_float4(lo[0], lo[1], lo[2], __uint_as_float(id));
      leaf[2 * (i >> 5) + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
    }
  }
  __syncthreads();
  if (wid != 0) return;
  for (int a = 0; a < 3; ++a) {
    lo[a] = s_lo[lane][a];
    hi[a] = s_hi[lane][a];
  }
  warp_min_max(lo, hi);
  id = __reduce_min_sync(0xffffffffu, s_id[lane]);
  if (lane == 0) {
    node[2 * blockIdx.x] = make_float4(lo[0], lo[1], lo[2], __uint_as_float(id));
    node[2 * blockIdx.x + 1] = make_float4(hi[0], hi[1], hi[2], 0.f);
  }
}

// binary32 squared distance in the specified order (no contraction)
__device__ __forceinline__ float dist2(float ax, float ay, float az, float bx, float by, float bz) {
  const float dx = fsub(bx, ax), dy = fsub(by, ay), dz = fsub(bz, az);
  return fadd(fadd(fmul(dx, dx), fmul(dy, dy)), fmul(dz, dz));
}

// A box as a query sees it: the bits of a lower bound of the squared distance
// from (x, y, z) to any point of it (the margin covers the roundings;
// non-negative, so the bits order as the values do), and the smallest index of
// its points.  A box that is not there or has been visited holds kKnnNone.
constexpr uint32_t kKnnNone = 0xffffffffu;
struct KnnBox {
  uint32_t gap, id;
  __device__ __forceinline__ KnnBox(const float4* __restrict__ box, bool there, float x, float y, float z)
      : gap(kKnnNone), id(kKnnNone) {
    if (!there) return;
    const float4 lo = __ldg(box), hi = __ldg(box + 1);
    const float gx = fmaxf(0.f, fmaxf(lo.x - x, x - hi.x));
    const float gy = fmaxf(0.f, fmaxf(lo.y - y, y - hi.y));
    const float gz = fmaxf(0.f, fmaxf(lo.z - z, z - hi.z));
    gap = __float_as_uint((gx * gx + gy * gy + gz * gz) * 0.99999f);
    id = __float_as_uint(lo.w);
  }
  // The lane whose box is the nearest that can hold a smaller key than the k-th
  // of `best` (wd: its distance bits), -1 if none can: at a gap of just wd, by a
  // smaller index.  (Coincident points, say a sensor's empty returns, all lie at
  // gap 0 = wd: without the indices each of them visited the leaves of all, 18 ms
  // with 50k of 102k points coincident, now 0.22.)
  __device__ __forceinline__ int nearest(uint32_t wd, unsigned long long best, int k) const {
    const uint32_t m = __reduce_min_sync(0xffffffffu, gap);
    if (m < wd) return __ffs(__ballot_sync(0xffffffffu, gap == m)) - 1;
    if (m > wd || m == kKnnNone) return -1;
    const uint32_t wid = __shfl_sync(0xffffffffu, static_cast<uint32_t>(best), k - 1);
    return __ffs(__ballot_sync(0xffffffffu, gap == m && id < wid)) - 1;
  }
};

// Compare-exchange with lane ^ j: the smaller key stays where `low` holds.
__device__ __forceinline__ void cas_lane(unsigned long long& v, int j, bool low) {
  const unsigned long long o = __shfl_xor_sync(0xffffffffu, v, j);
  v = (o < v) == low ? o : v;
}

constexpr int kKnnCta = 256;
// Candidates of a leaf taken one by one (about 14 instructions each) up to
// this many, by a bitonic sort and merge (about 190) beyond; 6 to 12 measured
// the same, 18 two percent slower.
constexpr int kKnnOneByOne = 12;

// One warp per query.  Lane l holds the l-th smallest key (distance bits,
// original index) of the points seen so far; `wd` is the k-th one's distance.
// The query's own leaf first, then the boxes that can still hold a closer
// point, nearest first, in its own node, the other nodes of its batch of 32
// and the other batches.  Bound by issue and by the latency of the box and
// point loads (L1 and L2 hits).  A query prunes with its own radius, and the
// k-th neighbour radii of a scan span 0.03 to 16 m: a CTA per 256 queries,
// pruning with the widest of its radii and lasting as long as its worst
// query, took 5.27 ms on the 102k points of a 128 x 1024 scan, this 0.136 ms
// (k = 20; the whole call 5.35 -> 0.191 ms, 51k points 2.73 -> 0.111 ms).
__global__ void __launch_bounds__(kKnnCta) k_ini_knn(const float4* __restrict__ sp, uint32_t n,
                                                     const float4* __restrict__ leaf_box, uint32_t n_leaf,
                                                     const float4* __restrict__ node_box, uint32_t n_node, int k,
                                                     int32_t* __restrict__ knn, int64_t* __restrict__ pairs) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  const int lane = threadIdx.x & 31;
  const uint32_t q = blockIdx.x * (kKnnCta / 32) + (threadIdx.x >> 5);
  if (q >= n) return;
  const float4 me = __ldg(sp + q);
  unsigned long long best = ~0ull;
  uint32_t wd = 0xffffffffu;   // distance bits of the k-th best (none yet)
  uint32_t evaluated = 0;
  const uint32_t leaf0 = q >> 5, node0 = q >> 10, batch0 = q >> 15;
  const uint32_t n_batch = (n_node + 31) / 32;
  bool first = true;   // on the way down to the query's own leaf
  for (uint32_t t = 0; t < n_batch; ++t) {
    const uint32_t batch = t == 0 ? batch0 : (t <= batch0 ? t - 1 : t);
    const uint32_t nd = 32 * batch + lane;
    KnnBox un(node_box + 2 * nd, nd < n_node, me.x, me.y, me.z);
    while (true) {
      const int a = first ? static_cast<int>(node0 & 31u) : un.nearest(wd, best, k);
      if (a < 0) break;
      if (lane == a) un.gap = kKnnNone;
      const uint32_t lf = 32 * (32 * batch + a) + lane;
      KnnBox ul(leaf_box + 2 * lf, lf < n_leaf, me.x, me.y, me.z);
      while (true) {
        const int b = first ? static_cast<int>(leaf0 & 31u) : ul.nearest(wd, best, k);
        if (b < 0) break;
        first = false;
        if (lane == b) ul.gap = kKnnNone;
        const uint32_t base = 32 * (32 * (32 * batch + a) + b);
        const uint32_t i = base + lane;
        evaluated += min(32u, n - base);
        uint32_t d = 0xffffffffu, id = 0xffffffffu;
        if (i < n) {
          const float4 p = __ldg(sp + i);
          d = __float_as_uint(dist2(me.x, me.y, me.z, p.x, p.y, p.z));
          id = __float_as_uint(p.w);
        }
        // (a distance equal to the k-th may still win by its index)
        uint32_t m = __ballot_sync(0xffffffffu, i < n && d <= wd);
        if (!m) continue;
        unsigned long long key = (static_cast<unsigned long long>(d) << 32) | id;
        if (__popc(m) <= kKnnOneByOne) {
          do {
            const unsigned long long x = __shfl_sync(0xffffffffu, key, __ffs(m) - 1);
            m &= m - 1;
            const uint32_t less = __ballot_sync(0xffffffffu, best < x);
            const unsigned long long up = __shfl_up_sync(0xffffffffu, best, 1);
            const int pos = __popc(less);
            best = lane < pos ? best : (lane == pos ? x : up);
          } while (m);
        } else {
          // candidates sorted descending, the smaller half of the two lists
          // (a bitonic sequence) merged
          if (!((m >> lane) & 1u)) key = ~0ull;
#pragma unroll
          for (int w = 2; w <= 32; w <<= 1)
#pragma unroll
            for (int j = w >> 1; j; j >>= 1) cas_lane(key, j, ((lane & j) == 0) == ((lane & w) != 0 && w < 32));
          best = key < best ? key : best;
#pragma unroll
          for (int j = 16; j; j >>= 1) cas_lane(best, j, (lane & j) == 0);
        }
        wd = static_cast<uint32_t>(__shfl_sync(0xffffffffu, best, k - 1) >> 32);
      }
    }
  }
  if (pairs && lane == 0) atomicAdd(reinterpret_cast<unsigned long long*>(pairs), static_cast<unsigned long long>(evaluated));
  if (lane < k) knn[static_cast<size_t>(__float_as_uint(me.w)) * k + lane] = static_cast<int32_t>(static_cast<uint32_t>(best));
}

// One cyclic-Jacobi rotation zeroing A[p][q] of the symmetric 3x3 A and
// accumulating it into V (Golub & Van Loan, the symmetric Schur
// decomposition of the 2x2 subproblem): A <- J^T A J, V <- V J.
__device__ __forceinline__ void jacobi_rotate(float (&A)[3][3], float (&V)[3][3], int p, int q) {
  const float apq = A[p][q];
  if (fabsf(apq) < 1e-36f) return;
  const float theta = (A[q][q] - A[p][p]) / (2.f * apq);
  float t;
  if (fabsf(theta) > 1e18f) {
    t = 0.5f / theta;
  } else {
    t = copysignf(1.f, theta) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
  }
  const float c = rsqrtf(t * t + 1.f), s = t * c;
  float B[3][3];
#pragma unroll
  for (int r = 0; r < 3; ++r) {   // B = A J
    B[r][p] = c * A[r][p] - s * A[r][q];
    B[r][q] = s * A[r][p] + c * A[r][q];
    B[r][3 - p - q] = A[r][3 - p - q];
  }
#pragma unroll
  for (int cidx = 0; cidx < 3; ++cidx) {   // A = J^T B
    A[p][cidx] = c * B[p][cidx] - s * B[q][cidx];
    A[q][cidx] = s * B[p][cidx] + c * B[q][cidx];
    A[3 - p - q][cidx] = B[3 - p - q][cidx];
  }
  A[p][q] = 0.f;
  A[q][p] = 0.f;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const float vp = V[r][p], vq = V[r][q];
    V[r][p] = c * vp - s * vq;
    V[r][q] = s * vp + c * vq;
  }
}

__global__ void __launch_bounds__(256) k_ini_frame(const float* __restrict__ pts, uint32_t n,
                                                   const int32_t* __restrict__ knn, IniParams P,
                                                   lgs_surfel_params_out out, float* __restrict__ lam,
                                                   float* __restrict__ conf) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float px = pts[3 * i], py = pts[3 * i + 1], pz = pts[3 * i + 2];
  const int k = P.k;
  // neighbour offsets from the point (exact for points within a factor of
  // two of each other, Sterbenz), their mean, and the centred second moments
  float mx = 0.f, my = 0.f, mz = 0.f;
  for (int t = 0; t < k; ++t) {
    const int j = knn[static_cast<size_t>(i) * k + t];
    mx += pts[3 * j] - px;
    my += pts[3 * j + 1] - py;
    mz += pts[3 * j + 2] - pz;
  }
  const float ik = 1.f / static_cast<float>(k);
  mx *= ik;
  my *= ik;
  mz *= ik;
  float cxx = 0.f, cxy = 0.f, cxz = 0.f, cyy = 0.f, cyz = 0.f, czz = 0.f;
  for (int t = 0; t < k; ++t) {
    const int j = knn[static_cast<size_t>(i) * k + t];
    const float dx = (pts[3 * j] - px) - mx, dy = (pts[3 * j + 1] - py) - my, dz = (pts[3 * j + 2] - pz) - mz;
    cxx += dx * dx;
    cxy += dx * dy;
    cxz += dx * dz;
    cyy += dy * dy;
    cyz += dy * dz;
    czz += dz * dz;
  }
  float A[3][3] = {{cxx * ik, cxy * ik, cxz * ik}, {cxy * ik, cyy * ik, cyz * ik}, {cxz * ik, cyz * ik, czz * ik}};
  float V[3][3] = {{1.f, 0.f, 0.f}, {0.f, 1.f, 0.f}, {0.f, 0.f, 1.f}};
  for (int sweep = 0; sweep < 6; ++sweep) {
    jacobi_rotate(A, V, 0, 1);
    jacobi_rotate(A, V, 0, 2);
    jacobi_rotate(A, V, 1, 2);
  }
  // eigenpairs in descending order
  float ev[3] = {A[0][0], A[1][1], A[2][2]};
  int o[3] = {0, 1, 2};
  if (ev[o[0]] < ev[o[1]]) { const int x = o[0]; o[0] = o[1]; o[1] = x; }
  if (ev[o[1]] < ev[o[2]]) { const int x = o[1]; o[1] = o[2]; o[2] = x; }
  if (ev[o[0]] < ev[o[1]]) { const int x = o[0]; o[0] = o[1]; o[1] = x; }
  const float l0 = fmaxf(ev[o[0]], 0.f), l1 = fmaxf(ev[o[1]], 0.f), l2 = fmaxf(ev[o[2]], 0.f);
  float3 e0 = make_float3(V[0][o[0]], V[1][o[0]], V[2][o[0]]);
  float3 nn = make_float3(V[0][o[2]], V[1][o[2]], V[2][o[2]]);
  // the normal turned toward the sensor (the origin of the sensor frame)
  if (nn.x * px + nn.y * py + nn.z * pz > 0.f) nn = make_float3(-nn.x, -nn.y, -nn.z);
  float nl = rsqrtf(nn.x * nn.x + nn.y * nn.y + nn.z * nn.z);
  nn = make_float3(nn.x * nl, nn.y * nl, nn.z * nl);
  const float en = e0.x * nn.x + e0.y * nn.y + e0.z * nn.z;
  e0 = make_float3(e0.x - en * nn.x, e0.y - en * nn.y, e0.z - en * nn.z);
  nl = rsqrtf(e0.x * e0.x + e0.y * e0.y + e0.z * e0.z);
  const float3 tu = make_float3(e0.x * nl, e0.y * nl, e0.z * nl);
  const float3 tv = make_float3(nn.y * tu.z - nn.z * tu.y, nn.z * tu.x - nn.x * tu.z, nn.x * tu.y - nn.y * tu.x);
  // range-adaptive scale: clip(kappa max(|p|, 1) sigma_tan, s_min, s_max)
  const float rng = sqrtf(px * px + py * py + pz * pz);
  const float sg0 = sqrtf(l0), sg1 = sqrtf(l1);
  const float t1 = sg0 > 0.f ? sg1 / sg0 : 1.f;   // sigma_tan = (1, sigma_1 / sigma_0)
  const float r = fmaxf(rng, 1.f);
  const float s0 = fminf(fmaxf(P.kappa * r, P.s_min), P.s_max);
  const float s1 = fminf(fmaxf(P.kappa * r * t1, P.s_min), P.s_max);
  // physics-based confidence and opacity
  const float cosv = fabsf(nn.x * px + nn.y * py + nn.z * pz) / rng;
  const float ramp = fminf(fmaxf((cosv - P.c0) / (1.f - P.c0 + P.eps), 0.f), 1.f);
  const float q = rng / P.r0;
  const float u = expf(-q * q) * ramp;
  const float alpha = P.alpha_min + (P.alpha_max - P.alpha_min) * u;
  // world frame: Rw = R [t_u t_v n]; quaternion by the largest of
  // 1 + tr, 1 + 2 R_ii - tr (Shepperd's rule), w >= 0
  float W[3][3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    W[a][0] = P.R[3 * a] * tu.x + P.R[3 * a + 1] * tu.y + P.R[3 * a + 2] * tu.z;
    W[a][1] = P.R[3 * a] * tv.x + P.R[3 * a + 1] * tv.y + P.R[3 * a + 2] * tv.z;
    W[a][2] = P.R[3 * a] * nn.x + P.R[3 * a + 1] * nn.y + P.R[3 * a + 2] * nn.z;
  }
  const float tr = W[0][0] + W[1][1] + W[2][2];
  const float c0 = 1.f + tr, c1 = 1.f + 2.f * W[0][0] - tr, c2 = 1.f + 2.f * W[1][1] - tr,
              c3 = 1.f + 2.f * W[2][2] - tr;
  float qw, qx, qy, qz;
  if (c0 >= c1 && c0 >= c2 && c0 >= c3) {
    const float h = 2.f * sqrtf(c0);
    qw = 0.25f * h; qx = (W[2][1] - W[1][2]) / h; qy = (W[0][2] - W[2][0]) / h; qz = (W[1][0] - W[0][1]) / h;
  } else if (c1 >= c2 && c1 >= c3) {
    const float h = 2.f * sqrtf(c1);
    qw = (W[2][1] - W[1][2]) / h; qx = 0.25f * h; qy = (W[0][1] + W[1][0]) / h; qz = (W[0][2] + W[2][0]) / h;
  } else if (c2 >= c3) {
    const float h = 2.f * sqrtf(c2);
    qw = (W[0][2] - W[2][0]) / h; qx = (W[0][1] + W[1][0]) / h; qy = 0.25f * h; qz = (W[1][2] + W[2][1]) / h;
  } else {
    const float h = 2.f * sqrtf(c3);
    qw = (W[1][0] - W[0][1]) / h; qx = (W[0][2] + W[2][0]) / h; qy = (W[1][2] + W[2][1]) / h; qz = 0.25f * h;
  }
  const float qn = rsqrtf(qw * qw + qx * qx + qy * qy + qz * qz) * (qw < 0.f ? -1.f : 1.f);
  out.quat[4 * i] = qw * qn;
  out.quat[4 * i + 1] = qx * qn;
  out.quat[4 * i + 2] = qy * qn;
  out.quat[4 * i + 3] = qz * qn;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    out.mean[3 * i + a] = P.R[3 * a] * px + P.R[3 * a + 1] * py + P.R[3 * a + 2] * pz + P.t[a];
  out.log_scale[2 * i] = logf(s0);
  out.log_scale[2 * i + 1] = logf(s1);
  out.opacity_logit[i] = logf(alpha / (1.f - alpha));
  lam[3 * i] = l0;
  lam[3 * i + 1] = l1;
  lam[3 * i + 2] = l2;
  conf[i] = u;
}

// Scratch: partial extents, the grid, the codes, the radix passes' counts
// and two buffers of (code, index) pairs, the points in cell order with their
// original index, leaf and node boxes.
struct IniLayout {
  size_t part, grid, code, hist, kv0, kv1, sp, leaf, node, total;
};

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

bool sort_wide(size_t n) { return n > (1u << 18); }   // 16 rounds of keys per sort CTA instead of 4

uint32_t sort_ctas(size_t n) {
  const size_t per = static_cast<size_t>(kIniSortCta) * (sort_wide(n) ? 16 : 4);
  return static_cast<uint32_t>((n + per - 1) / per);
}

IniLayout ini_layout(int64_t n) {
  IniLayout L{};
  const size_t N = static_cast<size_t>(n > 0 ? n : 1);
  size_t o = 0;
  auto take = [&](size_t bytes) { const size_t at = o; o = align256(o + bytes); return at; };
  L.part = take(kIniExtCtas * sizeof(IniBox));
  L.grid = take(sizeof(IniGrid));
  L.code = take(4 * N);
  L.hist = take(4 * static_cast<size_t>(kIniBins) * sort_ctas(N));
  L.kv0 = take(8 * N);
  L.kv1 = take(8 * N);
  L.sp = take(16 * N);
  L.leaf = take(32 * ((N + 31) / 32));
  L.node = take(32 * ((N + 1023) / 1024));
  L.total = o;
  return L;
}

// The points into cell order: three passes of count and scatter.
template <int R>
cudaError_t launch_order(const float* pts, uint32_t n, const IniLayout& L, char* b, cudaStream_t s) {
  const IniGrid* grid = reinterpret_cast<const IniGrid*>(b + L.grid);
  uint32_t* code = reinterpret_cast<uint32_t*>(b + L.code);
  uint32_t* hist = reinterpret_cast<uint32_t*>(b + L.hist);
  uint2* kv0 = reinterpret_cast<uint2*>(b + L.kv0);
  uint2* kv1 = reinterpret_cast<uint2*>(b + L.kv1);
  float4* sp = reinterpret_cast<float4*>(b + L.sp);
  const dim3 g(sort_ctas(n)), c(kIniSortCta);
  cudaError_t e = launch_dep(k_ini_count<R, true>, g, c, 0, s, pts, grid, code, nullptr, n, 0, hist);
  if (e == cudaSuccess) e = launch_dep(k_ini_scatter<R, true, false>, g, c, 0, s, code, nullptr, n, 0, hist, kv0, pts, sp);
  if (e == cudaSuccess) e = launch_dep(k_ini_count<R, false>, g, c, 0, s, pts, grid, code, kv0, n, kIniDigit, hist);
  if (e == cudaSuccess) e = launch_dep(k_ini_scatter<R, false, false>, g, c, 0, s, code, kv0, n, kIniDigit, hist, kv1, pts, sp);
  if (e == cudaSuccess) e = launch_dep(k_ini_count<R, false>, g, c, 0, s, pts, grid, code, kv1, n, 2 * kIniDigit, hist);
  if (e == cudaSuccess)
    e = launch_dep(k_ini_scatter<R, false, true>, g, c, 0, s, code, kv1, n, 2 * kIniDigit, hist, kv0, pts, sp);
  return e;
}

}  // namespace

size_t init_scratch_bytes(int64_t n) { return ini_layout(n).total; }

int64_t init_max_points() { return kIniMaxPoints; }

// partial extents, grid, three radix passes of count and scatter, boxes, k-NN,
// frame
int init_launches() { return 11; }

cudaError_t launch_keyframe_init(const float* pts, int64_t n64, const float pose[12], const lgs_init_params& p,
                                 void* scratch, int32_t* knn, const lgs_surfel_params_out& out, float* lam,
                                 float* conf, int64_t* pairs, cudaStream_t s) {
  const uint32_t n = static_cast<uint32_t>(n64);
  if (n == 0) return cudaSuccess;
  const IniLayout L = ini_layout(n);
  char* b = static_cast<char*>(scratch);
  IniBox* part = reinterpret_cast<IniBox*>(b + L.part);
  float4* sp = reinterpret_cast<float4*>(b + L.sp);
  float4* leaf = reinterpret_cast<float4*>(b + L.leaf);
  float4* node = reinterpret_cast<float4*>(b + L.node);
  const uint32_t n_part = std::min<uint32_t>((n + 255) / 256, kIniExtCtas);
  const uint32_t n_leaf = (n + 31) / 32, n_node = (n + 1023) / 1024;
  k_ini_part<<<n_part, 256, 0, s>>>(pts, n, part);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess)
    e = launch_dep(k_ini_grid, dim3(1), dim3(32), 0, s, part, n_part, reinterpret_cast<IniGrid*>(b + L.grid));
  if (e == cudaSuccess) e = sort_wide(n) ? launch_order<16>(pts, n, L, b, s) : launch_order<4>(pts, n, L, b, s);
  if (e == cudaSuccess) e = launch_dep(k_ini_boxes, dim3(n_node), dim3(1024), 0, s, sp, n, leaf, node);
  if (e == cudaSuccess)
    e = launch_dep(k_ini_knn, dim3((n + kKnnCta / 32 - 1) / (kKnnCta / 32)), dim3(kKnnCta), 0, s, sp, n, leaf, n_leaf,
                   node, n_node, p.k, knn, pairs);
  if (e != cudaSuccess) return e;
  IniParams P;
  for (int a = 0; a < 3; ++a) {
    for (int b = 0; b < 3; ++b) P.R[3 * a + b] = pose[4 * a + b];
    P.t[a] = pose[4 * a + 3];
  }
  P.kappa = p.kappa;
  P.s_min = p.s_min;
  P.s_max = p.s_max;
  P.r0 = p.r0;
  P.c0 = p.c0;
  P.eps = p.eps;
  P.alpha_min = p.alpha_min;
  P.alpha_max = p.alpha_max;
  P.k = p.k;
  return launch_dep(k_ini_frame, dim3((n + 255) / 256), dim3(256), 0, s, pts, n, knn, P, out, lam, conf);
}

}  // namespace lgs
