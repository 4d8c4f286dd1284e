// lgs_raster.cu -- per-tile front-to-back compositing (forward) and its
// reverse-order adjoint (backward) for the spherical surfel rasterizer.
//
// One CTA renders one angular tile (tile_h x tile_w pixels, one thread per
// pixel).  The tile's depth-ordered list is streamed through shared memory in
// batches of BATCH records (64 B each, gathered by item id); every thread
// walks the batch for its own ray.  Pixels stop once T (1 - a) would drop
// below 1e-4; a warp whose lanes have all stopped skips the batch, and the
// CTA leaves when every pixel has stopped.
//
// The backward re-evaluates the same records per tile in reverse list order
// (no per-pixel surfel lists are stored): the transmittance before each
// contributor is recovered as T_k = T_{k+1} / (1 - a_k) from T_final, and the
// suffix sum S = sum_{j>k} w_j (g . c_j) gives dL/da_k = T_k (g . c_k) -
// S / (1 - a_k).  Per entry the warp reduces its 15 geometric gradients with a
// butterfly reduce-scatter (16 shuffles), 15 lanes add them into a shared
// per-batch accumulator, and the CTA flushes one atomic add per (surfel,
// component) into the per-item gradient buffer.
#include <cstddef>
#include <cuda_runtime.h>

#include "lgs_internal.cuh"

namespace lgs {

constexpr int kMaxTileThreads = 256;
// Per-item gradient moments written by the backward.  With the unclamped
// opacity derivative g = alpha G dL/da of a contribution (0 where a is
// clamped), its offset (u, v) in the plane, ct = (dL/dt) / (n.d) and the
// direct normal term w sg gS_n, every surfel gradient is a fixed combination
// of their sums over the contributions (k_preprocess_bwd forms it):
//   [0] g  [1] u g  [2] v g  [3] u^2 g  [4] v^2 g  [5] u v g
//   [6] ct  [7] ct u  [8] ct v  [9..11] w sg gS_n
// because dL/du = -u g, dL/dv = -v g and the intersection offset inside the
// plane is u s_u t_u + v s_v t_v.
constexpr int kGrad = 12;

// The 12 moments of one valid contribution with transmittance Tk before it
// and suffix S (the sum over the later contributors of w (g.c)), added into v.
__device__ __forceinline__ void moments(const Eval& E, const float4& r0, float Tk, float S, float iom, float gA,
                                        float gSt, float gSx, float gSy, float gSz, float (&v)[16]) {
  const float sg = E.den > 0.f ? -1.f : 1.f;
  const float gc = gA + gSt * E.t + sg * (gSx * r0.x + gSy * r0.y + gSz * r0.z);
  const float w = E.a * Tk;
  const float dLda = Tk * gc - S * iom;
  const float g = E.araw < 0.99f ? E.araw * dLda : 0.f;
  const float ug = E.u * g, vg = E.v * g;
  const float ct = fmaf(w, gSt, -fmaf(ug, E.ud, vg * E.vd)) * E.rden;
  const float wsg = w * sg;
  v[0] += g;
  v[1] += ug;
  v[2] += vg;
  v[3] += E.u * ug;
  v[4] += E.v * vg;
  v[5] += E.u * vg;
  v[6] += ct;
  v[7] += ct * E.u;
  v[8] += ct * E.v;
  v[9] += wsg * gSx;
  v[10] += wsg * gSy;
  v[11] += wsg * gSz;
}

// Reverse-order step of one valid contribution: updates the transmittance T
// (before it) and the suffix S, and adds its 12 moments into v (the same
// arithmetic as moments(), with S updated in place).
__device__ __forceinline__ void contrib_moments(const Eval& E, const float4& r0, float gA, float gSt, float gSx,
                                                float gSy, float gSz, float& T, float& S, float (&v)[16]) {
  const float iom = rcp_ftz(1.0f - E.a);
  const float Tk = T * iom;
  const float sg = E.den > 0.f ? -1.f : 1.f;
  const float gc = gA + gSt * E.t + sg * (gSx * r0.x + gSy * r0.y + gSz * r0.z);
  const float w = E.a * Tk;
  const float dLda = Tk * gc - S * iom;
  S = fmaf(w, gc, S);
  T = Tk;
  const float g = E.araw < 0.99f ? E.araw * dLda : 0.f;
  const float ug = E.u * g, vg = E.v * g;
  const float ct = fmaf(w, gSt, -fmaf(ug, E.ud, vg * E.vd)) * E.rden;
  const float wsg = w * sg;
  v[0] += g;
  v[1] += ug;
  v[2] += vg;
  v[3] += E.u * ug;
  v[4] += E.v * vg;
  v[5] += E.u * vg;
  v[6] += ct;
  v[7] += ct * E.u;
  v[8] += ct * E.v;
  v[9] += wsg * gSx;
  v[10] += wsg * gSy;
  v[11] += wsg * gSz;
}

struct TileCtx {
  int f;
  int r, c;
  bool inside;
  uint32_t start, end;
  int64_t pix;
  int HW;
};

__device__ __forceinline__ TileCtx tile_ctx(const Desc& D, uint32_t tile, const uint2* __restrict__ ranges,
                                            int vt) {
  TileCtx t;
  t.f = frame_of_tile(D, tile);
  const FrameDev& F = D.f[t.f];
  const int lt = static_cast<int>(tile - F.tile_base);
  const int ti = lt / F.ntc, tj = lt - ti * F.ntc;
  int lr, lc;
  pixel_of_thread(F, vt, lr, lc);
  t.r = ti * F.th + lr;
  t.c = tj * F.tw + lc;
  t.inside = t.r < F.H && t.c < F.W;
  t.pix = static_cast<int64_t>(t.r) * F.W + t.c;
  t.HW = F.H * F.W;
  const uint2 rg = ranges[tile];
  t.start = rg.x;
  t.end = rg.y;
  return t;
}

// Work item of the CTA: its own tile, or (persistent mode) the next entry of
// the longest-first order claimed through an atomic counter.
__device__ __forceinline__ bool next_tile(bool persistent, const uint32_t* __restrict__ order, uint32_t n_tiles,
                                          unsigned int* counter, uint32_t& tile, int iter) {
  if (!persistent) {
    tile = blockIdx.x;
    return iter == 0;
  }
  __shared__ uint32_t s_tile;
  __syncthreads();
  if (threadIdx.x == 0) s_tile = atomicAdd(counter, 1u);
  __syncthreads();
  const uint32_t k = s_tile;
  if (k >= n_tiles) return false;
  tile = order ? order[k] : k;
  return true;
}

// The batch entries whose pixel box meets the warp's pixel block, in list
// order: 32 boxes tested per step (one per lane) and compacted with a ballot.
// Returns the count (uniform over the warp).
__device__ __forceinline__ int warp_list(const float4* s_box, int nb, const WarpBox& wb, uint16_t* list) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  int cnt = 0;
  for (int base = 0; base < nb; base += 32) {
    const int j = base + lane;
    const bool hit = j < nb && box_hits(s_box[j], wb);
    const uint32_t m = __ballot_sync(0xffffffffu, hit);
    if (hit) list[cnt + __popc(m & lt)] = static_cast<uint16_t>(j);
    cnt += __popc(m);
  }
  __syncwarp();
  return cnt;
}

// ---------------------------------------------------------------------------
// Forward
// ---------------------------------------------------------------------------
template <int BATCH>
__global__ void __launch_bounds__(kMaxTileThreads)
    k_fwd(const Desc* __restrict__ D, const uint2* __restrict__ ranges, const uint32_t* __restrict__ pv,
          const float4* __restrict__ rec, const float4* __restrict__ box, const uint32_t* __restrict__ order,
          Status* __restrict__ st, int persistent) {
  __shared__ float4 s_r0[BATCH], s_r1[BATCH], s_r2[BATCH], s_box[BATCH];
  __shared__ float s_al[BATCH];
  __shared__ uint16_t s_list[kMaxTileThreads / 32][BATCH];
  const int nthr = blockDim.x;
  const int tid = threadIdx.x, wid = tid >> 5;
  uint32_t tile;
  uint32_t evals = 0, contrib = 0, alg = 0;
  for (int iter = 0; next_tile(persistent, order, D->n_tiles, &st->work_counter, tile, iter); ++iter) {
    const TileCtx tc = tile_ctx(*D, tile, ranges, static_cast<int>(threadIdx.x));
    if (tc.end - tc.start > kLongList) continue;   // the long-list kernels' tile
    const FrameDev& F = D->f[tc.f];
    const WarpBox wb = warp_box(tc.inside, tc.r, tc.c, F.W);
    float dx = 0.f, dy = 0.f, dz = 0.f;
    if (tc.inside) pixel_ray(F, tc.r, tc.c, dx, dy, dz);
    float T = 1.0f, A = 0.0f, St = 0.0f, Sx = 0.0f, Sy = 0.0f, Sz = 0.0f;
    int last = 0, stop_at = -1;
    bool done = !tc.inside;
    for (uint32_t b0 = tc.start; b0 < tc.end; b0 += BATCH) {
      if (__syncthreads_and(done)) break;
      const int nb = static_cast<int>(min(static_cast<uint32_t>(BATCH), tc.end - b0));
      for (int j = tid; j < nb; j += nthr) {
        const uint32_t item = pv[b0 + j];
        const float4* rp = rec + 4 * static_cast<int64_t>(item);
        s_r0[j] = rp[0];
        s_r1[j] = rp[1];
        s_r2[j] = rp[2];
        s_al[j] = rp[3].x;
        s_box[j] = box[item];
      }
      __syncthreads();
      int cnt = 0;
      if (!__all_sync(0xffffffffu, done)) cnt = warp_list(s_box, nb, wb, s_list[wid]);
      if (!done) {
        for (int k = 0; k < cnt; k += 2) {
          const int jj[2] = {s_list[wid][k], k + 1 < cnt ? s_list[wid][k + 1] : s_list[wid][k]};
          Eval ee[2];
#pragma unroll
          for (int q = 0; q < 2; ++q) eval_pair(s_r0[jj[q]], s_r1[jj[q]], s_r2[jj[q]], s_al[jj[q]], dx, dy, dz, ee[q]);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            if (done || k + q >= cnt) break;
            const int j = jj[q];
            const Eval& e = ee[q];
            ++evals;
            if (!e.valid) continue;
            const float Tn = __fmul_rn(T, __fsub_rn(1.0f, e.a));
            if (Tn < 1e-4f) {
              done = true;
              stop_at = static_cast<int>(b0 - tc.start) + j + 1;
              break;
            }
            const float w = e.a * T;
            const float ws = e.den > 0.f ? -w : w;
            A += w;
            St = fmaf(w, e.t, St);
            Sx = fmaf(ws, s_r0[j].x, Sx);
            Sy = fmaf(ws, s_r0[j].y, Sy);
            Sz = fmaf(ws, s_r0[j].z, Sz);
            T = Tn;
            last = static_cast<int>(b0 - tc.start) + j + 1;
            ++contrib;
          }
          if (done) break;
        }
      }
    }
    if (tc.inside) {
      F.A[tc.pix] = A;
      F.St[tc.pix] = St;
      F.Sn[tc.pix] = Sx;
      F.Sn[tc.HW + tc.pix] = Sy;
      F.Sn[2 * static_cast<int64_t>(tc.HW) + tc.pix] = Sz;
      F.Tf[tc.pix] = T;
      F.nc[tc.pix] = last;
      alg += stop_at >= 0 ? static_cast<uint32_t>(stop_at) : tc.end - tc.start;
    }
  }
  unsigned long long ev = evals, co = contrib;
  for (int o = 16; o > 0; o >>= 1) {
    ev += __shfl_xor_sync(0xffffffffu, ev, o);
    co += __shfl_xor_sync(0xffffffffu, co, o);
  }
  unsigned long long al = alg;
  for (int o = 16; o > 0; o >>= 1) al += __shfl_xor_sync(0xffffffffu, al, o);
  if ((tid & 31) == 0 && ev) atomicAdd(&st->evals_fwd, ev);
  if ((tid & 31) == 0 && co) atomicAdd(&st->contrib_fwd, co);
  if ((tid & 31) == 0 && al) atomicAdd(&st->alg_fwd, al);
}

// ---------------------------------------------------------------------------
// Backward
// ---------------------------------------------------------------------------
// Butterfly reduce-scatter of 16 values over the warp: afterwards lane L holds
// in v[0] the warp sum of value index 8 b4 + 4 b3 + 2 b2 + b1 (bits of L).
__device__ __forceinline__ void warp_reduce16(float (&v)[16], int lane) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const bool hi = lane & 16;
    const float send = hi ? v[i] : v[i + 8];
    const float keep = hi ? v[i + 8] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool hi = lane & 8;
    const float send = hi ? v[i] : v[i + 4];
    const float keep = hi ? v[i + 4] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool hi = lane & 4;
    const float send = hi ? v[i] : v[i + 2];
    const float keep = hi ? v[i + 2] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  {
    const bool hi = lane & 2;
    const float send = hi ? v[0] : v[1];
    const float keep = hi ? v[1] : v[0];
    v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
}

template <int BATCH>
__global__ void __launch_bounds__(kMaxTileThreads)
    k_bwd(const Desc* __restrict__ D, const uint2* __restrict__ ranges, const uint32_t* __restrict__ pv,
          const float4* __restrict__ rec, const float4* __restrict__ box, float* __restrict__ g13,
          const uint32_t* __restrict__ order, Status* __restrict__ st, int persistent) {
  __shared__ float4 s_r0[BATCH], s_r1[BATCH], s_r2[BATCH], s_r3[BATCH], s_box[BATCH];
  __shared__ uint16_t s_list[kMaxTileThreads / 32][BATCH];
  __shared__ uint32_t s_item[BATCH];
  __shared__ float s_g[kGrad][BATCH];
  __shared__ int s_max;
  const int nthr = blockDim.x;
  const int tid = threadIdx.x, lane = tid & 31;
  const int gidx = 8 * ((lane >> 4) & 1) + 4 * ((lane >> 3) & 1) + 2 * ((lane >> 2) & 1) + ((lane >> 1) & 1);
  const bool writer = ((lane & 1) == 0) && gidx < kGrad;
  uint32_t tile;
  uint32_t evals = 0, contrib = 0;
  for (int iter = 0; next_tile(persistent, order, D->n_tiles, &st->work_counter2, tile, iter); ++iter) {
    const TileCtx tc = tile_ctx(*D, tile, ranges, static_cast<int>(threadIdx.x));
    if (tc.end - tc.start > kLongList) continue;   // the long-list kernels' tile
    const FrameDev& F = D->f[tc.f];
    const WarpBox wb = warp_box(tc.inside, tc.r, tc.c, F.W);
    float dx = 0.f, dy = 0.f, dz = 0.f;
    float T = 1.f, gA = 0.f, gSt = 0.f, gSx = 0.f, gSy = 0.f, gSz = 0.f;
    int nc = 0;
    if (tc.inside) {
      pixel_ray(F, tc.r, tc.c, dx, dy, dz);
      T = F.Tf[tc.pix];
      nc = F.nc[tc.pix];
      gA = F.gA[tc.pix];
      gSt = F.gSt[tc.pix];
      gSx = F.gSn[tc.pix];
      gSy = F.gSn[tc.HW + tc.pix];
      gSz = F.gSn[2 * static_cast<int64_t>(tc.HW) + tc.pix];
    }
    if (tid == 0) s_max = 0;
    __syncthreads();
    if (nc > 0) atomicMax(&s_max, nc);
    __syncthreads();
    // n_contrib comes from the caller: never walk past the tile's list
    const uint32_t len = tc.end - tc.start;
    const uint32_t stop = tc.start + min(static_cast<uint32_t>(s_max), len);
    float S = 0.f;
    for (uint32_t bend = stop; bend > tc.start;) {
      const uint32_t b0 = bend - tc.start > static_cast<uint32_t>(BATCH) ? bend - BATCH : tc.start;
      const int nb = static_cast<int>(bend - b0);
      __syncthreads();
      for (int j = tid; j < nb; j += nthr) {
        const uint32_t item = pv[b0 + j];
        s_item[j] = item;
        const float4* rp = rec + 4 * static_cast<int64_t>(item);
        s_r0[j] = rp[0];
        s_r1[j] = rp[1];
        s_r2[j] = rp[2];
        s_r3[j] = rp[3];
        s_box[j] = box[item];
#pragma unroll
        for (int c = 0; c < kGrad; ++c) s_g[c][j] = 0.f;
      }
      __syncthreads();
      const int cnt = warp_list(s_box, nb, wb, s_list[tid >> 5]);
      for (int kk = cnt - 1; kk >= 0; --kk) {
        const int j = s_list[tid >> 5][kk];
        const int k = static_cast<int>(b0 - tc.start) + j;
        float v[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = 0.f;
        bool valid = false;
        if (k < nc) {
          const float4 r0 = s_r0[j];
          const float alpha = s_r3[j].x;
          Eval e;
          eval_pair(r0, s_r1[j], s_r2[j], alpha, dx, dy, dz, e);
          ++evals;
          valid = e.valid;
          if (valid) {
            ++contrib;
            contrib_moments(e, r0, gA, gSt, gSx, gSy, gSz, T, S, v);
          }
        }
        if (__any_sync(0xffffffffu, valid)) {
          warp_reduce16(v, lane);
          if (writer) atomicAdd(&s_g[gidx][j], v[0]);
        }
      }
      __syncthreads();
      for (int j = tid; j < nb; j += nthr) {
        float* gp = g13 + 16 * static_cast<int64_t>(s_item[j]);
#pragma unroll
        for (int c = 0; c < kGrad; ++c) {
          const float x = s_g[c][j];
          if (x != 0.f) atomicAdd(gp + c, x);
        }
      }
      bend = b0;
    }
  }
  unsigned long long ev = evals, co = contrib;
  for (int o = 16; o > 0; o >>= 1) {
    ev += __shfl_xor_sync(0xffffffffu, ev, o);
    co += __shfl_xor_sync(0xffffffffu, co, o);
  }
  if ((tid & 31) == 0 && ev) atomicAdd(&st->evals_bwd, ev);
  if ((tid & 31) == 0 && co) atomicAdd(&st->contrib_bwd, co);
}

// ---------------------------------------------------------------------------
// Warp-independent walk (batch = 0)
// ---------------------------------------------------------------------------
// Each warp culls and composites the tile list on its own: 32 entries per
// step (one pixel box per lane, compacted with a ballot), records of the hits
// read by the whole warp from L1 (broadcast loads; a tile's records are
// shared by its warps through L1 instead of shared memory), the next hit's
// record fetched while the current one is composited.  No CTA barrier sits in
// the loop: a warp leaves when its own pixels have stopped, and the backward
// walks only up to its own pixels' last contributor.  The per-pixel
// arithmetic and order are those of the batched kernels (results are
// bit-identical in the forward).
struct Rec {
  float4 r0, r1, r2, r3;
};

__device__ __forceinline__ Rec load_rec(const float4* __restrict__ rec, uint32_t item) {
  const float4* rp = rec + 4 * static_cast<int64_t>(item);
  Rec r;
  r.r0 = __ldg(rp);
  r.r1 = __ldg(rp + 1);
  r.r2 = __ldg(rp + 2);
  r.r3 = __ldg(rp + 3);
  return r;
}

// G hits per step: their records are fetched and evaluated together (G
// independent chains for the scheduler), then composited in list order.
template <int G>
__global__ void __launch_bounds__(kMaxTileThreads)
    k_fwd_w(const Desc* __restrict__ D, const uint2* __restrict__ ranges, const uint32_t* __restrict__ pv,
            const float4* __restrict__ rec, const float4* __restrict__ box, const uint32_t* __restrict__ order,
            Status* __restrict__ st, int persistent) {
  const int lane = threadIdx.x & 31;
  uint32_t tile;
  uint32_t evals = 0, contrib = 0, alg = 0;
  for (int iter = 0; next_tile(persistent, order, D->n_tiles, &st->work_counter, tile, iter); ++iter) {
    const TileCtx tc = tile_ctx(*D, tile, ranges, static_cast<int>(threadIdx.x));
    if (tc.end - tc.start > kLongList) continue;   // the long-list kernels' tile
    const FrameDev& F = D->f[tc.f];
    const WarpBox wb = warp_box(tc.inside, tc.r, tc.c, F.W);
    float dx = 0.f, dy = 0.f, dz = 0.f;
    if (tc.inside) pixel_ray(F, tc.r, tc.c, dx, dy, dz);
    float T = 1.0f, A = 0.0f, St = 0.0f, Sx = 0.0f, Sy = 0.0f, Sz = 0.0f;
    int last = 0, stop_at = -1;
    bool done = !tc.inside;
    for (uint32_t base = tc.start; base < tc.end; base += 32) {
      if (__all_sync(0xffffffffu, done)) break;
      const uint32_t j = base + lane;
      uint32_t item = 0;
      bool hit = false;
      if (j < tc.end) {
        item = __ldg(pv + j);
        hit = box_hits(__ldg(box + item), wb);
      }
      uint32_t m = __ballot_sync(0xffffffffu, hit);
      while (m) {
        int bq[G];
        float4 r0[G], r1[G], r2[G];
        float al[G];
#pragma unroll
        for (int q = 0; q < G; ++q) {
          bq[q] = m ? __ffs(m) - 1 : -1;
          m &= m - 1;
          if (bq[q] >= 0) {
            const float4* rp = rec + 4 * static_cast<int64_t>(__shfl_sync(0xffffffffu, item, bq[q]));
            r0[q] = __ldg(rp);
            r1[q] = __ldg(rp + 1);
            r2[q] = __ldg(rp + 2);
            al[q] = __ldg(reinterpret_cast<const float*>(rp + 3));
          }
        }
        Eval e[G];
#pragma unroll
        for (int q = 0; q < G; ++q)
          if (bq[q] >= 0) eval_pair(r0[q], r1[q], r2[q], al[q], dx, dy, dz, e[q]);
#pragma unroll
        for (int q = 0; q < G; ++q) {
          if (bq[q] < 0 || done) continue;
          ++evals;
          if (!e[q].valid) continue;
          const float Tn = __fmul_rn(T, __fsub_rn(1.0f, e[q].a));
          if (Tn < 1e-4f) {
            done = true;
            stop_at = static_cast<int>(base - tc.start) + bq[q] + 1;
            continue;
          }
          const float w = e[q].a * T;
          const float ws = e[q].den > 0.f ? -w : w;
          A += w;
          St = fmaf(w, e[q].t, St);
          Sx = fmaf(ws, r0[q].x, Sx);
          Sy = fmaf(ws, r0[q].y, Sy);
          Sz = fmaf(ws, r0[q].z, Sz);
          T = Tn;
          last = static_cast<int>(base - tc.start) + bq[q] + 1;
          ++contrib;
        }
        if (__all_sync(0xffffffffu, done)) break;
      }
    }
    if (tc.inside) {
      F.A[tc.pix] = A;
      F.St[tc.pix] = St;
      F.Sn[tc.pix] = Sx;
      F.Sn[tc.HW + tc.pix] = Sy;
      F.Sn[2 * static_cast<int64_t>(tc.HW) + tc.pix] = Sz;
      F.Tf[tc.pix] = T;
      F.nc[tc.pix] = last;
      alg += stop_at >= 0 ? static_cast<uint32_t>(stop_at) : tc.end - tc.start;
    }
  }
  unsigned long long ev = evals, co = contrib;
  for (int o = 16; o > 0; o >>= 1) {
    ev += __shfl_xor_sync(0xffffffffu, ev, o);
    co += __shfl_xor_sync(0xffffffffu, co, o);
  }
  unsigned long long al = alg;
  for (int o = 16; o > 0; o >>= 1) al += __shfl_xor_sync(0xffffffffu, al, o);
  if (lane == 0 && ev) atomicAdd(&st->evals_fwd, ev);
  if (lane == 0 && co) atomicAdd(&st->contrib_fwd, co);
  if (lane == 0 && al) atomicAdd(&st->alg_fwd, al);
}

template <int G>
__global__ void __launch_bounds__(kMaxTileThreads)
    k_bwd_w(const Desc* __restrict__ D, const uint2* __restrict__ ranges, const uint32_t* __restrict__ pv,
            const float4* __restrict__ rec, const float4* __restrict__ box, float* __restrict__ g13,
            const uint32_t* __restrict__ order, Status* __restrict__ st, int persistent) {
  const int lane = threadIdx.x & 31;
  const int gidx = 8 * ((lane >> 4) & 1) + 4 * ((lane >> 3) & 1) + 2 * ((lane >> 2) & 1) + ((lane >> 1) & 1);
  const bool writer = ((lane & 1) == 0) && gidx < kGrad;
  uint32_t tile;
  uint32_t evals = 0, contrib = 0;
  for (int iter = 0; next_tile(persistent, order, D->n_tiles, &st->work_counter2, tile, iter); ++iter) {
    const TileCtx tc = tile_ctx(*D, tile, ranges, static_cast<int>(threadIdx.x));
    if (tc.end - tc.start > kLongList) continue;   // the long-list kernels' tile
    const FrameDev& F = D->f[tc.f];
    const WarpBox wb = warp_box(tc.inside, tc.r, tc.c, F.W);
    float dx = 0.f, dy = 0.f, dz = 0.f;
    float T = 1.f, gA = 0.f, gSt = 0.f, gSx = 0.f, gSy = 0.f, gSz = 0.f;
    int nc = 0;
    if (tc.inside) {
      pixel_ray(F, tc.r, tc.c, dx, dy, dz);
      T = F.Tf[tc.pix];
      nc = F.nc[tc.pix];
      gA = F.gA[tc.pix];
      gSt = F.gSt[tc.pix];
      gSx = F.gSn[tc.pix];
      gSy = F.gSn[tc.HW + tc.pix];
      gSz = F.gSn[2 * static_cast<int64_t>(tc.HW) + tc.pix];
    }
    // n_contrib comes from the caller: never walk past the tile's list
    const uint32_t len = tc.end - tc.start;
    const uint32_t stop = min(static_cast<uint32_t>(__reduce_max_sync(0xffffffffu, nc > 0 ? nc : 0)), len);
    float S = 0.f;
    for (int c0 = static_cast<int>((stop + 31) / 32) - 1; c0 >= 0; --c0) {
      const uint32_t k0 = 32u * c0;
      uint32_t item = 0;
      bool hit = false;
      if (k0 + lane < stop) {
        item = __ldg(pv + tc.start + k0 + lane);
        hit = box_hits(__ldg(box + item), wb);
      }
      uint32_t m = __ballot_sync(0xffffffffu, hit);
      while (m) {
        int bq[G];
        uint32_t itq[G];
        float4 r0[G], r1[G], r2[G];
        float al[G];
#pragma unroll
        for (int q = 0; q < G; ++q) {
          bq[q] = m ? 31 - __clz(m) : -1;
          if (bq[q] >= 0) {
            m &= ~(1u << bq[q]);
            itq[q] = __shfl_sync(0xffffffffu, item, bq[q]);
            const float4* rp = rec + 4 * static_cast<int64_t>(itq[q]);
            r0[q] = __ldg(rp);
            r1[q] = __ldg(rp + 1);
            r2[q] = __ldg(rp + 2);
            al[q] = __ldg(reinterpret_cast<const float*>(rp + 3));
          }
        }
        Eval e[G];
        bool in[G];
#pragma unroll
        for (int q = 0; q < G; ++q) {
          in[q] = bq[q] >= 0 && static_cast<int>(k0 + bq[q]) < nc;
          if (in[q]) eval_pair(r0[q], r1[q], r2[q], al[q], dx, dy, dz, e[q]);
        }
#pragma unroll
        for (int q = 0; q < G; ++q) {
          if (bq[q] < 0) break;
          const bool valid = in[q] && e[q].valid;
          evals += in[q];
          float v[16];
#pragma unroll
          for (int c = 0; c < 16; ++c) v[c] = 0.f;
          if (valid) {
            ++contrib;
            contrib_moments(e[q], r0[q], gA, gSt, gSx, gSy, gSz, T, S, v);
          }
          if (__any_sync(0xffffffffu, valid)) {
            warp_reduce16(v, lane);
            if (writer && v[0] != 0.f) atomicAdd(g13 + 16 * static_cast<int64_t>(itq[q]) + gidx, v[0]);
          }
        }
      }
    }
  }
  unsigned long long ev = evals, co = contrib;
  for (int o = 16; o > 0; o >>= 1) {
    ev += __shfl_xor_sync(0xffffffffu, ev, o);
    co += __shfl_xor_sync(0xffffffffu, co, o);
  }
  if (lane == 0 && ev) atomicAdd(&st->evals_bwd, ev);
  if (lane == 0 && co) atomicAdd(&st->contrib_bwd, co);
}

// ---------------------------------------------------------------------------
// Reduce-scatter of the 12 gradient moments of one (warp, entry) over the
// warp: 15 shuffles for 12 values.
// ---------------------------------------------------------------------------
// Reduce-scatter of 12 values over the warp.  Afterwards the warp sum of
// value 6 b4 + 3 b3 + b2 is held by the lanes with (lane & 3) == 0 and that
// of value 6 b4 + 3 b3 + 2 by the lanes with (lane & 7) == 1 (b4, b3, b2 the
// lane's bits); returns the lane's value and sets idx (-1: not a writer).
__device__ __forceinline__ float warp_reduce12(const float (&v)[12], int lane, int& idx) {
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  float w[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const float send = b4 ? v[i] : v[i + 6];
    const float keep = b4 ? v[i + 6] : v[i];
    w[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
  float x[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float send = b3 ? w[i] : w[i + 3];
    const float keep = b3 ? w[i + 3] : w[i];
    x[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  float y0, y2;
  {
    const float send = b2 ? x[0] : x[1];
    const float keep = b2 ? x[1] : x[0];
    y0 = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    y2 = x[2] + __shfl_xor_sync(0xffffffffu, x[2], 4);
  }
  y0 += __shfl_xor_sync(0xffffffffu, y0, 2);
  y2 += __shfl_xor_sync(0xffffffffu, y2, 2);
  y0 += __shfl_xor_sync(0xffffffffu, y0, 1);
  y2 += __shfl_xor_sync(0xffffffffu, y2, 1);
  const int base = (b4 ? 6 : 0) + (b3 ? 3 : 0);
  const bool first = (lane & 3) == 0;
  idx = first ? base + (b2 ? 1 : 0) : ((lane & 7) == 1 ? base + 2 : -1);
  return first ? y0 : y2;
}

// ---------------------------------------------------------------------------
// Shared-memory walk (group 16): each warp walks its tile list in chunks of
// 32 entries; the records of the chunk's hits are staged in the warp's own
// shared-memory slots (one 48-B record per lane) and read back with broadcast
// loads, so a hit costs no shuffle, no 64-bit address arithmetic and no
// global load on the critical path.  No CTA barrier: warps proceed alone.
// ---------------------------------------------------------------------------
struct WarpRecs {
  float4 r0[32], r1[32], r2[32];
  float al[32];
};

__device__ __forceinline__ void stage_hit(const float4* __restrict__ rec, uint32_t item, WarpRecs& s, int lane) {
  const float4* rp = rec + 4 * static_cast<int64_t>(item);
  s.r0[lane] = __ldg(rp);
  s.r1[lane] = __ldg(rp + 1);
  s.r2[lane] = __ldg(rp + 2);
  s.al[lane] = __ldg(reinterpret_cast<const float*>(rp + 3));
}

// Image-loss epilogue of the forward kernels: the pixel's terms from its
// composited values still in registers (no re-read of the planes), its
// upstream gradient planes written, the terms' fixed-point values summed over
// the warp and added to the frame's loss sums (one atomic per term and warp).
struct LossEpi {
  lgs_loss_params P;
  int* ctot;                     // mask counts [frame][2], complete before the forward
  unsigned long long* acc;       // fixed-point sums [frame][4], then [maps] of the regulariser
  float* out;                    // loss vector, written by the forward's last CTA
};

__device__ __forceinline__ void loss_epilogue(const Desc& D, const LossEpi& L, int f, bool inside, int64_t pix,
                                              int HW, float A, float St, float Sx, float Sy, float Sz) {
  long long ld = 0, la = 0, ln = 0;
  if (inside) {
    const FrameDev& F = D.f[f];
    const int nd = __ldcg(L.ctot + 2 * f), nn = __ldcg(L.ctot + 2 * f + 1);
    const float scale = 1.0f / static_cast<float>(D.m[F.map].n_frames);
    const float ind = nd > 0 ? 1.0f / static_cast<float>(nd) : 0.f;
    const float inn = nn > 0 ? 1.0f / static_cast<float>(nn) : 0.f;
    float g[5];
    pixel_image_loss(F.D[pix], A, St, F.Ng[pix], F.Ng[HW + pix], F.Ng[2 * static_cast<int64_t>(HW) + pix], Sx, Sy,
                     Sz, scale, ind, inn, L.P, g, ld, la, ln);
    F.oA[pix] = g[0];
    F.oSt[pix] = g[1];
    F.oSn[pix] = g[2];
    F.oSn[HW + pix] = g[3];
    F.oSn[2 * static_cast<int64_t>(HW) + pix] = g[4];
  }
  for (int o = 16; o > 0; o >>= 1) {
    ld += __shfl_xor_sync(0xffffffffu, ld, o);
    la += __shfl_xor_sync(0xffffffffu, la, o);
    ln += __shfl_xor_sync(0xffffffffu, ln, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (ld) atomicAdd(L.acc + 4 * f, static_cast<unsigned long long>(ld));
    if (la) atomicAdd(L.acc + 4 * f + 1, static_cast<unsigned long long>(la));
    if (ln) atomicAdd(L.acc + 4 * f + 2, static_cast<unsigned long long>(ln));
  }
}

__device__ __forceinline__ uint32_t warp_claim(unsigned int* counter) {
  uint32_t id = 0;
  if ((threadIdx.x & 31) == 0) id = atomicAdd(counter, 1u);
  return __shfl_sync(0xffffffffu, id, 0);
}

// A warp that finds no work left counts itself done; the last of `total` resets
// the work and done counters to zero for the next launch on the stream.
__device__ __forceinline__ void long_finish(unsigned int* counter, unsigned int* done, unsigned int total) {
  if ((threadIdx.x & 31) == 0) {
    __threadfence();
    if (atomicAdd(done, 1u) == total - 1) {
      *counter = 0u;
      *done = 0u;
    }
  }
}

// ---------------------------------------------------------------------------
// Long lists (more than kLongList entries) in the forward
// ---------------------------------------------------------------------------
// A tile with a very long list (a far horizon seen along a street: tens of
// thousands of entries, few of which any pixel composites) would make its
// warps walk the list alone while the rest of the frame is done.  Two steps:
//  (1) k_long_masks: the list is cut into segments of kSeg entries, and warps
//      claim (segment, pixel block) items: the warp finds which entries are
//      valid at which of its 32 pixels and writes the window masks.  Items are
//      claimed segment by segment over all long lists, so that a pixel's first
//      segments are usually done before its later ones start: a segment behind
//      one whose entries alone stop the pixel is skipped.
//  (2) k_fwd_long, one warp per pixel: the 32 lanes take the entries of a
//      window that the masks name; the transmittance before each is T times a
//      multiplicative scan of (1 - a) over the lanes, the early stop is the
//      first lane whose T (1 - a) falls below 1e-4, and the composited sums
//      are warp reductions.  Windows without a valid entry are skipped.
// The lists' box tests and evaluations, shared by 32 pixels in (1), were the
// bulk of (2) when it walked every window of the list itself with a box test
// per (pixel, entry): 8 keyframes of a 1M map (17.9 M long entries) 3.5 ms, now
// 0.53 + 0.87; 6 maps (26.8 M) 4.8 ms, now 0.52 + 0.60.
// The products and sums associate differently from the per-tile walk (same
// values to a few ulps), and exactly as they did without step (1).
constexpr int kSegSlots = 5;   // a segment's sums of w, w t, w n'(3)

struct SegBuf {
  const uint2* item;       // [segments] (long list, segment), segment by segment
  const uint32_t* longt;   // [long lists] tile
  const uint32_t* sbase;   // [tiles] first segment of a long list
  float* sum;              // [segments][kSegSlots][tile pixels]
  uint32_t* dead;          // [long lists][tile pixels] first segment known to stop the pixel (~0: none)
};

// Step (1) takes a pixel for stopped a little below the threshold: its product
// of (1 - a) associates differently from step (2)'s.
constexpr float kSurelyStopped = 0.99e-4f;

// The pixels of a 4 x 8 block (rows r0 .. r0 + 3, columns cmid - 3.5 .. cmid +
// 3.5, one bit each in lane order) inside a culling box.  A box that nearly
// wraps around the frame takes every column (its distance is formed for the
// block's centre, so a pixel of the block could be nearer the other way round).
__device__ __forceinline__ uint32_t block_cover(const float4& b, float r0, float cmid, float W, float inv_W) {
  const int lo = max(static_cast<int>(ceilf(b.x - r0)), 0), hi = min(static_cast<int>(floorf(b.y - r0)), 3);
  if (lo > hi) return 0u;
  uint32_t cols = 0xffu;
  if (b.w < 0.5f * W - 8.0f) {
    float d = b.z - cmid;
    d -= W * rintf(d * inv_W);
    const int cl = max(static_cast<int>(ceilf(fmaxf(d - b.w, -4.0f) + 3.5f)), 0);
    const int ch = min(static_cast<int>(floorf(fminf(d + b.w, 4.0f) + 3.5f)), 7);
    if (cl > ch) return 0u;
    cols = (2u << ch) - (1u << cl);
  }
  const uint32_t rows = 0x01010101u & (0xffffffffu << (8 * lo)) & (0xffffffffu >> (8 * (3 - hi)));
  return cols * rows;
}

// Transpose of a 32 x 32 bit matrix, one row per lane: bit j of lane i becomes
// bit i of lane j.
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane) {
  uint32_t m = 0x0000ffffu;
#pragma unroll
  for (int k = 16; k; k >>= 1) {
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, k);
    x = (lane & k) ? (x & ~m) | ((y & ~m) >> k) : (x & m) | ((y & m) << k);
    m ^= m << (k >> 1);
  }
  return x;
}

// The pixels of a warp and the entries that may be valid at them.  Lane i holds
// entry i of a window (box b; ok: there is one); candidates() returns the
// entries to evaluate at the lane's pixel, one bit each, and sets hit where the
// lane's entry is one of some pixel's.
template <bool BLOCK48>
struct WarpPixels;

// 4 x 8 blocks (pixel_of_thread): every lane finds the pixels inside its
// entry's box, and a transpose gives every pixel its entries.
template <>
struct WarpPixels<true> {
  float r0, cmid, W, inv_W;
  __device__ __forceinline__ WarpPixels(const FrameDev& F, const TileCtx& tc, int lane)
      : r0(static_cast<float>(tc.r - (lane >> 3))),
        cmid(static_cast<float>(tc.c - (lane & 7)) + 3.5f),
        W(static_cast<float>(F.W)),
        inv_W(1.0f / static_cast<float>(F.W)) {}
  __device__ __forceinline__ uint32_t candidates(const float4& b, bool ok, int lane, bool& hit) const {
    const uint32_t cover = ok ? block_cover(b, r0, cmid, W, inv_W) : 0u;
    hit = cover != 0u;
    return warp_transpose(cover, lane);
  }
};

// Any other shape: every pixel takes the entries whose box meets the warp's
// pixels.  (Each box tested again per pixel, four shuffles and ten instructions
// for every such entry, cost more than the evaluations it spared: the street
// frame's forward, 200k surfels, 238, 220 and 289 us with tiles of 2 x 16, 16 x 4
// and 1 x 64 pixels, against 144, 150 and 191.)
template <>
struct WarpPixels<false> {
  WarpBox wb;
  __device__ __forceinline__ WarpPixels(const FrameDev& F, const TileCtx& tc, int)
      : wb(warp_box(tc.inside, tc.r, tc.c, F.W)) {}
  __device__ __forceinline__ uint32_t candidates(const float4& b, bool ok, int, bool& hit) const {
    hit = ok && box_hits(b, wb);
    return __ballot_sync(0xffffffffu, hit);
  }
};

// Candidates a lane evaluates together per step of the shared-memory forward
// (street frame, bin and forward: 1 169.9 us, 2 167.3, 3 165.6; its step and
// 8 keyframes of a 1M map: 357.8, 347.0, 350.2 us and 6.31, 6.13, 6.10 ms).
// Every lane takes its own next candidates (street frame: 17 per window and
// warp at most over the lanes, where the warp took all 21 hits together; the
// forward 115 -> 111 us).
constexpr int FWD_HITS = 2;

// Step (1) of the long lists: warps claim (segment, block) items.
template <bool BLOCK48>
__global__ void __launch_bounds__(256, 3)
    k_long_masks(const Desc* __restrict__ Dp, const uint2* __restrict__ ranges, const uint32_t* __restrict__ pv,
                 const float4* __restrict__ rec, const float4* __restrict__ box, Status* __restrict__ st,
                 const uint32_t* __restrict__ cbase, float* __restrict__ ckpt, uint32_t* __restrict__ cmask,
                 uint32_t* __restrict__ bwm, SegBuf seg) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ WarpRecs s_w[8];
  const Desc& D = *Dp;
  const int lane = threadIdx.x & 31;
  WarpRecs& sw = s_w[threadIdx.x >> 5];
  const int npx = D.th * D.tw;
  const uint32_t blocks = static_cast<uint32_t>(npx) >> 5;
  const uint32_t n_items = st->n_segs * blocks;
  if (n_items == 0) return;
  uint32_t evals = 0;
  while (true) {
    const uint32_t id = warp_claim(&st->seg_counter);
    if (id >= n_items) break;
    const uint2 it = __ldg(seg.item + id / blocks);
    const uint32_t li = it.x, sg = it.y, tile = __ldg(seg.longt + li);
    const int vt = static_cast<int>(id % blocks) * 32 + lane;
    // (step (2) takes the maximum over the block's pixels; a block outside the
    // frame has none, and the backward's queues read its word all the same)
    if (sg == 0 && lane == 0) bwm[tile * blocks + id % blocks] = 0u;
    const TileCtx tc = tile_ctx(D, tile, ranges, vt);
    uint32_t* dead = seg.dead + static_cast<int64_t>(li) * npx + vt;
    bool done = !tc.inside || __ldcg(dead) < sg;
    if (__all_sync(0xffffffffu, done)) continue;
    const FrameDev& F = D.f[tc.f];
    const WarpPixels<BLOCK48> bb(F, tc, lane);
    float dx = 0.f, dy = 0.f, dz = 0.f;
    if (tc.inside) pixel_ray(F, tc.r, tc.c, dx, dy, dz);
    const uint32_t first = tc.start + sg * kSeg, end = min(first + kSeg, tc.end);
    // the checkpoints and the segment's sums start empty (step (2) writes the
    // chunks and segments in which the pixel composites something)
    const int64_t cb = static_cast<int64_t>(cbase[tile]);
    for (uint32_t c = sg * kSegChunks; c * kChunk < end - tc.start; ++c)
#pragma unroll
      for (int k = 0; k < kCkptSlots; ++k) ckpt[((cb + c) * kCkptSlots + k) * npx + vt] = 0.f;
#pragma unroll
    for (int k = 0; k < kSegSlots; ++k)
      seg.sum[((static_cast<int64_t>(__ldg(seg.sbase + tile)) + sg) * kSegSlots + k) * npx + vt] = 0.f;
    float T = 1.0f;
    uint32_t item_nx = first + 32 + lane < end ? __ldg(pv + first + 32 + lane) : 0u;
    uint32_t item_cur = first + lane < end ? __ldg(pv + first + lane) : 0u;
    float4 box_cur = first + lane < end ? __ldg(box + item_cur) : make_float4(0.f, 0.f, 0.f, 0.f);
    for (uint32_t base = first; base < end; base += 32) {
      if (__all_sync(0xffffffffu, done)) break;
      uint32_t* mword = cmask + (cb * 4 + (base - tc.start) / 32) * npx + vt;
      const uint32_t j = base + lane;
      const uint32_t item = item_cur;
      const float4 bx = box_cur;
      item_cur = item_nx;
      box_cur = j + 32 < end ? __ldg(box + item_nx) : make_float4(0.f, 0.f, 0.f, 0.f);
      item_nx = j + 64 < end ? __ldg(pv + j + 64) : 0u;
      bool hit;
      uint32_t m = bb.candidates(bx, j < end, lane, hit);
      if (done) m = 0u;
      uint32_t cbits = 0;
      if (__any_sync(0xffffffffu, m)) {
        evals += __popc(m);
        const int idle = __ffs(__ballot_sync(0xffffffffu, hit)) - 1;
        __syncwarp();
        if (hit) stage_hit(rec, item, sw, lane);
        __syncwarp();
        do {
          int bq[FWD_HITS];
          bool on[FWD_HITS];
          Eval e[FWD_HITS];
#pragma unroll
          for (int q = 0; q < FWD_HITS; ++q) {
            on[q] = m != 0u;
            bq[q] = on[q] ? __ffs(m) - 1 : idle;
            m &= m - 1;
            eval_pair(sw.r0[bq[q]], sw.r1[bq[q]], sw.r2[bq[q]], sw.al[bq[q]], dx, dy, dz, e[q]);
          }
#pragma unroll
          for (int q = 0; q < FWD_HITS; ++q) {
            const bool ok = on[q] && e[q].valid;
            cbits |= ok ? 1u << bq[q] : 0u;
            T *= ok ? 1.0f - e[q].a : 1.0f;
          }
        } while (__any_sync(0xffffffffu, m));
        if (!done && T < kSurelyStopped) {
          done = true;
          atomicMin(dead, sg);
        }
      }
      *mword = cbits;
    }
  }
  long_finish(&st->seg_counter, &st->seg_done, gridDim.x * (blockDim.x >> 5));
  unsigned long long ev = evals;
  for (int o = 16; o > 0; o >>= 1) ev += __shfl_xor_sync(0xffffffffu, ev, o);
  if (lane == 0 && ev) atomicAdd(&st->evals_fwd, ev);
}

// The tiles with short lists: every CTA its own, or persistent ones claiming
// them.  The long lists were composited before; with LOSS the CTA that finishes
// last writes the loss vector.
// At most 72 registers: 14 CTAs of an 8 x 8 tile (64 threads) per SM, so
// the 2048 tiles of a 128 x 1024 frame fit in one wave on 152 SMs (75
// registers leave 72 tiles for a second wave).
template <bool LOSS, bool BLOCK48>
__global__ void __maxnreg__(72)
    k_fwd_s(const Desc* __restrict__ D, const uint2* __restrict__ ranges, const uint32_t* __restrict__ pv,
            const float4* __restrict__ rec, const float4* __restrict__ box, const uint32_t* __restrict__ order,
            Status* __restrict__ st, int persistent, const uint32_t* __restrict__ cbase, float* __restrict__ ckpt,
            uint32_t* __restrict__ cmask, uint32_t* __restrict__ bwm, LossEpi loss) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ WarpRecs s_w[kMaxTileThreads / 32];
  const int lane = threadIdx.x & 31;
  WarpRecs& sw = s_w[threadIdx.x >> 5];
  uint32_t tile;
  uint32_t evals = 0, contrib = 0, alg = 0;
  for (int iter = 0; next_tile(persistent, order, D->n_tiles, &st->work_counter, tile, iter); ++iter) {
    const TileCtx tc = tile_ctx(*D, tile, ranges, static_cast<int>(threadIdx.x));
    if (tc.end - tc.start > kLongList) continue;   // k_fwd_long's tile
    const FrameDev& F = D->f[tc.f];
    const WarpPixels<BLOCK48> bb(F, tc, lane);
    float dx = 0.f, dy = 0.f, dz = 0.f;
    if (tc.inside) pixel_ray(F, tc.r, tc.c, dx, dy, dz);
    float T = 1.0f, A = 0.0f, St = 0.0f, Sx = 0.0f, Sy = 0.0f, Sz = 0.0f;
    int last = 0, stop_at = -1;
    bool done = !tc.inside;
    // checkpoint of the backward chunks: this chunk's own sums, written with
    // T at every chunk end (the chunk holding the end of the walk included)
    float cA = 0.f, cSt = 0.f, cSx = 0.f, cSy = 0.f, cSz = 0.f;
    uint32_t chunk = 0;
    const int npx = static_cast<int>(blockDim.x);
    const auto checkpoint = [&]() {
      float* o = ckpt + (static_cast<int64_t>(cbase[tile] + chunk) * kCkptSlots) * npx + threadIdx.x;
      o[0] = T;
      o[npx] = cA;
      o[2 * npx] = cSt;
      o[3 * npx] = cSx;
      o[4 * npx] = cSy;
      o[5 * npx] = cSz;
      cA = cSt = cSx = cSy = cSz = 0.f;
    };
    // software pipeline over the windows: the list entry two windows ahead
    // and the culling box one window ahead are loaded while this window is
    // composited (entry, box and record would otherwise be a chain of
    // dependent round trips per window)
    uint32_t item_nx = tc.start + 32 + lane < tc.end ? __ldg(pv + tc.start + 32 + lane) : 0u;
    uint32_t item_cur = tc.start + lane < tc.end ? __ldg(pv + tc.start + lane) : 0u;
    float4 box_cur = tc.start + lane < tc.end ? __ldg(box + item_cur) : make_float4(0.f, 0.f, 0.f, 0.f);
    for (uint32_t base = tc.start; base < tc.end; base += 32) {
      if (base - tc.start >= (chunk + 1) * kChunk) {
        checkpoint();
        ++chunk;
      }
      if (__all_sync(0xffffffffu, done)) break;
      // the pixel's composited entries of this window, one bit each, for the
      // chunked backward (every window the warp walks gets its word)
      uint32_t* mword = cmask + (static_cast<int64_t>(cbase[tile]) * 4 + (base - tc.start) / 32) * npx + threadIdx.x;
      const uint32_t j = base + lane;
      const uint32_t item = item_cur;
      const float4 bx = box_cur;
      item_cur = item_nx;
      box_cur = j + 32 < tc.end ? __ldg(box + item_nx) : make_float4(0.f, 0.f, 0.f, 0.f);
      item_nx = j + 64 < tc.end ? __ldg(pv + j + 64) : 0u;
      // the pixel's candidates of the window, one bit per entry
      bool hit;
      uint32_t m = bb.candidates(bx, j < tc.end, lane, hit);
      if (done) m = 0u;
      if (!__any_sync(0xffffffffu, m)) {
        *mword = 0u;
        continue;
      }
      const uint32_t m_cand = m;
      // a lane without a candidate evaluates a staged one with weight 0 (its
      // record is finite; an unused slot may hold anything)
      const int idle = __ffs(__ballot_sync(0xffffffffu, hit)) - 1;
      __syncwarp();
      if (hit) stage_hit(rec, item, sw, lane);
      __syncwarp();
      const int k0 = static_cast<int>(base - tc.start) + 1;
      uint32_t cbits = 0;
      // composite one evaluated hit without branches: lanes that are done or
      // see an invalid pair add zeros and keep T (t and the weight are zeroed
      // first, so no inf or NaN of a rejected pair reaches the sums)
      const auto composite = [&](const Eval& e, const float4& r0, int bq) {
        const bool act = !done && e.valid;
        const float Tn = __fmul_rn(T, __fsub_rn(1.0f, e.a));
        const bool stop = act && Tn < 1e-4f;
        const bool comp = act && !(Tn < 1e-4f);
        const float w = comp ? e.a * T : 0.0f;
        const float tt = comp ? e.t : 0.0f;
        const float ws = e.den > 0.f ? -w : w;
        A += w;
        St = fmaf(w, tt, St);
        Sx = fmaf(ws, r0.x, Sx);
        Sy = fmaf(ws, r0.y, Sy);
        Sz = fmaf(ws, r0.z, Sz);
        cA += w;
        cSt = fmaf(w, tt, cSt);
        cSx = fmaf(ws, r0.x, cSx);
        cSy = fmaf(ws, r0.y, cSy);
        cSz = fmaf(ws, r0.z, cSz);
        T = comp ? Tn : T;
        cbits |= comp ? 1u << bq : 0u;
        stop_at = stop ? k0 + bq : stop_at;
        done = done || stop;
      };
      // every lane takes its own next FWD_HITS candidates: their evaluations
      // are independent (instruction-level parallelism), the composites
      // follow in list order
      do {
        int bq[FWD_HITS];
        bool on[FWD_HITS];
        float4 r0q[FWD_HITS];
        Eval eq[FWD_HITS];
#pragma unroll
        for (int q = 0; q < FWD_HITS; ++q) {
          on[q] = m != 0u;
          bq[q] = on[q] ? __ffs(m) - 1 : idle;
          m &= m - 1;
          r0q[q] = sw.r0[bq[q]];
          eval_pair(r0q[q], sw.r1[bq[q]], sw.r2[bq[q]], sw.al[bq[q]], dx, dy, dz, eq[q]);
          eq[q].valid = eq[q].valid && on[q];
        }
#pragma unroll
        for (int q = 0; q < FWD_HITS; ++q) composite(eq[q], r0q[q], bq[q]);
        if (done) m = 0u;
      } while (__any_sync(0xffffffffu, m));
      *mword = cbits;
      // the window's statistics from its bits: composited pairs, the last
      // one, and the candidates evaluated before the pixel stopped (through
      // the stop entry when it stopped in this window)
      if (cbits) last = k0 + (31 - __clz(cbits));
      contrib += __popc(cbits);
      evals += __popc(stop_at >= k0 ? m_cand & (0xffffffffu >> (31 - (stop_at - k0))) : m_cand);
    }
    if (tc.end > tc.start) checkpoint();
    if (tc.inside) {
      F.A[tc.pix] = A;
      F.St[tc.pix] = St;
      F.Sn[tc.pix] = Sx;
      F.Sn[tc.HW + tc.pix] = Sy;
      F.Sn[2 * static_cast<int64_t>(tc.HW) + tc.pix] = Sz;
      F.Tf[tc.pix] = T;
      F.nc[tc.pix] = last;
      alg += stop_at >= 0 ? static_cast<uint32_t>(stop_at) : tc.end - tc.start;
    }
    // the block's largest n_contrib: the backward's chunks of this block end there
    const uint32_t wmax = __reduce_max_sync(0xffffffffu, static_cast<uint32_t>(last));
    if (lane == 0) bwm[tile * (blockDim.x >> 5) + (threadIdx.x >> 5)] = wmax;
    if (LOSS) loss_epilogue(*D, loss, tc.f, tc.inside, tc.pix, tc.HW, A, St, Sx, Sy, Sz);
  }
  unsigned long long ev = evals, co = contrib;
  for (int o = 16; o > 0; o >>= 1) {
    ev += __shfl_xor_sync(0xffffffffu, ev, o);
    co += __shfl_xor_sync(0xffffffffu, co, o);
  }
  unsigned long long al = alg;
  for (int o = 16; o > 0; o >>= 1) al += __shfl_xor_sync(0xffffffffu, al, o);
  if (lane == 0 && ev) atomicAdd(&st->evals_fwd, ev);
  if (lane == 0 && co) atomicAdd(&st->contrib_fwd, co);
  if (lane == 0 && al) atomicAdd(&st->alg_fwd, al);
  if (LOSS) {
    // every pixel's epilogue has added its terms when the last CTA is done
    // (the regulariser was summed and the long lists composited before): it
    // writes the loss vector
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&st->loss_ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (s_last && threadIdx.x < 32) finish_loss_vector(*D, loss.P, loss.ctot, loss.acc, loss.out, st);
  }
}

// Thread of the per-tile forward that holds tile pixel (lr, lc) (the inverse
// of pixel_of_thread): the chunk checkpoints and window masks are laid out by
// it.
__device__ __forceinline__ int thread_of_pixel(const FrameDev& F, int lr, int lc) {
  if ((F.tw & 7) == 0 && (F.th & 3) == 0) {
    const int wpr = F.tw >> 3;
    return ((((lr >> 2) * wpr) + (lc >> 3)) << 5) | ((lr & 3) << 3) | (lc & 7);
  }
  return lr * F.tw + lc;
}

struct LongPix {
  const FrameDev* F;
  int r, c;
  bool inside;
  uint32_t start, end, tile, li;
  int64_t pix;
  int HW;
  int vt;   // the pixel's thread in the per-tile layout (checkpoints, masks)
};

__device__ __forceinline__ bool long_item(const Desc& D, const uint2* __restrict__ ranges,
                                          const uint32_t* __restrict__ longt, uint32_t n_long, uint32_t id,
                                          LongPix& p) {
  const uint32_t tp = static_cast<uint32_t>(D.th * D.tw);
  const uint32_t gi = id / tp, k = id - gi * tp;
  if (gi >= n_long) return false;
  const uint32_t tile = longt[gi];
  const int f = frame_of_tile(D, tile);
  const FrameDev& F = D.f[f];
  const int lt = static_cast<int>(tile - F.tile_base);
  const int ti = lt / F.ntc, tj = lt - ti * F.ntc;
  p.F = &F;
  p.tile = tile;
  p.li = gi;
  p.vt = thread_of_pixel(F, static_cast<int>(k) / F.tw, static_cast<int>(k) % F.tw);
  p.r = ti * F.th + static_cast<int>(k) / F.tw;
  p.c = tj * F.tw + static_cast<int>(k) % F.tw;
  p.inside = p.r < F.H && p.c < F.W;
  p.pix = static_cast<int64_t>(p.r) * F.W + p.c;
  p.HW = F.H * F.W;
  const uint2 rg = ranges[tile];
  p.start = rg.x;
  p.end = rg.y;
  return true;
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// Step (2) of the long lists: one warp per pixel (see above).  Software
// pipeline over the non-empty windows: the entries two ahead and the records
// one ahead are loaded while a window is composited.
template <bool LOSS>
__global__ void __launch_bounds__(256, 3) k_fwd_long(const Desc* __restrict__ D, const uint2* __restrict__ ranges,
                                                  const uint32_t* __restrict__ pv, const float4* __restrict__ rec,
                                                  Status* __restrict__ st, const uint32_t* __restrict__ cbase,
                                                  float* __restrict__ ckpt, const uint32_t* __restrict__ cmask,
                                                  uint32_t* __restrict__ bwm, LossEpi loss, SegBuf seg) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  const int lane = threadIdx.x & 31;
  const uint32_t n_long = st->n_long;
  if (n_long == 0) return;
  const int npx = D->th * D->tw;
  uint32_t contrib = 0, alg = 0;
  LongPix P;
  while (long_item(*D, ranges, seg.longt, n_long, warp_claim(&st->long_counter_fwd), P)) {
    if (!P.inside) continue;
    const FrameDev& F = *P.F;
    float dx, dy, dz;
    pixel_ray(F, P.r, P.c, dx, dy, dz);
    float T = 1.f, A = 0.f, St = 0.f, Sx = 0.f, Sy = 0.f, Sz = 0.f;
    int last = 0, stop_at = -1;
    const int64_t cb = static_cast<int64_t>(cbase[P.tile]), sb = static_cast<int64_t>(seg.sbase[P.tile]);
    const uint32_t* words = cmask + cb * 4 * npx + P.vt;
    const uint32_t n_win = (P.end - P.start + 31) / 32;
    // the chunked backward's inputs: T and the chunk's own sums at the end of
    // every chunk in which the pixel composites something, and the segments'
    // sums (the others are zero: step (1))
    float cA = 0.f, cSt = 0.f, cSx = 0.f, cSy = 0.f, cSz = 0.f;
    float g[kSegSlots] = {0.f, 0.f, 0.f, 0.f, 0.f};
    uint32_t chunk = ~0u;   // the chunk being composited
    const auto close_chunk = [&](uint32_t next) {
      if (chunk == ~0u) return;
      const float v[kSegSlots] = {warp_sum(cA), warp_sum(cSt), warp_sum(cSx), warp_sum(cSy), warp_sum(cSz)};
      if (lane == 0) {
        float* o = ckpt + ((cb + chunk) * kCkptSlots) * npx + P.vt;
        o[0] = T;
#pragma unroll
        for (int q = 0; q < kSegSlots; ++q) o[(q + 1) * npx] = v[q];
      }
      cA = cSt = cSx = cSy = cSz = 0.f;
#pragma unroll
      for (int q = 0; q < kSegSlots; ++q) g[q] += v[q];
      const uint32_t sg = chunk / kSegChunks;
      if (next != ~0u && next / kSegChunks == sg) return;
#pragma unroll
      for (int q = 0; q < kSegSlots; ++q) {
        if (lane == 0) seg.sum[((sb + sg) * kSegSlots + q) * npx + P.vt] = g[q];
        g[q] = 0.f;
      }
    };
    // the non-empty windows in order, found 32 mask words at a time (words
    // past the pixel's stop are not set; the walk ends before it uses them)
    uint32_t w0 = 0, word = static_cast<uint32_t>(lane) < n_win ? __ldg(words + static_cast<int64_t>(lane) * npx) : 0u;
    uint32_t word_nx = 32u + lane < n_win ? __ldg(words + static_cast<int64_t>(32 + lane) * npx) : 0u;
    uint32_t nz = __ballot_sync(0xffffffffu, word != 0u);
    const auto advance = [&](uint32_t& win, uint32_t& bits) -> bool {
      while (!nz) {
        w0 += 32;
        if (w0 >= n_win) return false;
        word = word_nx;
        word_nx = w0 + 32 + lane < n_win ? __ldg(words + static_cast<int64_t>(w0 + 32 + lane) * npx) : 0u;
        nz = __ballot_sync(0xffffffffu, word != 0u);
      }
      const int b = __ffs(nz) - 1;
      nz &= nz - 1;
      bits = __shfl_sync(0xffffffffu, word, b);
      win = w0 + b;
      return true;
    };
    const auto entry = [&](bool on, uint32_t win, uint32_t bits) -> uint32_t {
      const uint32_t j = P.start + 32 * win + lane;
      return on && ((bits >> lane) & 1u) && j < P.end ? __ldg(pv + j) : ~0u;
    };
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const auto load = [&](uint32_t item, float4& r0, float4& r1, float4& r2, float& al) {
      const float4* rp = rec + 4 * static_cast<int64_t>(item);
      const bool on = item != ~0u;
      r0 = on ? __ldg(rp) : zero;
      r1 = on ? __ldg(rp + 1) : zero;
      r2 = on ? __ldg(rp + 2) : zero;
      al = on ? __ldg(reinterpret_cast<const float*>(rp + 3)) : 0.f;
    };
    uint32_t win = 0, bits = 0, win1 = 0, bits1 = 0, win2 = 0, bits2 = 0;
    bool on = advance(win, bits);
    uint32_t item = entry(on, win, bits);
    bool on1 = on && advance(win1, bits1);
    uint32_t item1 = entry(on1, win1, bits1);
    float4 r0, r1, r2;
    float al;
    load(item, r0, r1, r2, al);
    while (on) {
      const bool on2 = on1 && advance(win2, bits2);
      const uint32_t item2 = entry(on2, win2, bits2);
      float4 q0, q1, q2;
      float ql;
      load(item1, q0, q1, q2, ql);
      if (win / 4 != chunk) {
        close_chunk(win / 4);
        chunk = win / 4;
      }
      const bool valid = item != ~0u;
      Eval e;
      eval_pair(r0, r1, r2, al, dx, dy, dz, e);
      // P_j = prod_{i <= j} (1 - a_i) over the valid lanes
      float Pj = valid ? __fsub_rn(1.0f, e.a) : 1.0f;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_up_sync(0xffffffffu, Pj, o);
        if (lane >= o) Pj *= y;
      }
      float Pex = __shfl_up_sync(0xffffffffu, Pj, 1);
      if (lane == 0) Pex = 1.0f;
      const uint32_t sm = __ballot_sync(0xffffffffu, valid && T * Pj < 1e-4f);
      const int fs = sm ? __ffs(sm) - 1 : 32;
      const bool inc = valid && lane < fs;
      const float w = inc ? e.a * (T * Pex) : 0.f;
      const float ws = valid && e.den > 0.f ? -w : w;
      // every lane sums its own entries' terms; the pixel's totals are the
      // warp sums of these after the walk
      A += w;
      if (inc) St = fmaf(w, e.t, St);
      Sx = fmaf(ws, r0.x, Sx);
      Sy = fmaf(ws, r0.y, Sy);
      Sz = fmaf(ws, r0.z, Sz);
      cA += w;
      if (inc) cSt = fmaf(w, e.t, cSt);
      cSx = fmaf(ws, r0.x, cSx);
      cSy = fmaf(ws, r0.y, cSy);
      cSz = fmaf(ws, r0.z, cSz);
      contrib += inc;
      const uint32_t im = __ballot_sync(0xffffffffu, inc);
      if (im) last = static_cast<int>(32 * win) + (31 - __clz(im)) + 1;
      T *= __shfl_sync(0xffffffffu, fs < 32 ? Pex : Pj, fs < 32 ? fs : 31);
      if (sm) {
        stop_at = static_cast<int>(32 * win) + fs + 1;
        break;
      }
      on = on1;
      win = win1;
      bits = bits1;
      item = item1;
      on1 = on2;
      win1 = win2;
      bits1 = bits2;
      item1 = item2;
      r0 = q0;
      r1 = q1;
      r2 = q2;
      al = ql;
    }
    close_chunk(~0u);
    A = warp_sum(A);
    St = warp_sum(St);
    Sx = warp_sum(Sx);
    Sy = warp_sum(Sy);
    Sz = warp_sum(Sz);
    if (lane == 0) {
      F.A[P.pix] = A;
      F.St[P.pix] = St;
      F.Sn[P.pix] = Sx;
      F.Sn[P.HW + P.pix] = Sy;
      F.Sn[2 * static_cast<int64_t>(P.HW) + P.pix] = Sz;
      F.Tf[P.pix] = T;
      F.nc[P.pix] = last;
      alg += stop_at >= 0 ? static_cast<uint32_t>(stop_at) : P.end - P.start;
      seg.dead[static_cast<int64_t>(P.li) * npx + P.vt] = ~0u;   // for the next forward
      if (last) atomicMax(bwm + (static_cast<int64_t>(P.tile) * npx + P.vt) / 32, static_cast<uint32_t>(last));
    }
    // the warp holds one pixel: lane 0 alone takes its loss terms
    if (LOSS) loss_epilogue(*D, loss, static_cast<int>(P.F - D->f), lane == 0, P.pix, P.HW, A, St, Sx, Sy, Sz);
  }
  long_finish(&st->long_counter_fwd, &st->long_done_fwd, gridDim.x * (blockDim.x >> 5));
  unsigned long long co = contrib, al64 = alg;
  for (int o = 16; o > 0; o >>= 1) co += __shfl_xor_sync(0xffffffffu, co, o);
  if (lane == 0 && co) atomicAdd(&st->contrib_fwd, co);
  if (lane == 0 && al64) atomicAdd(&st->alg_fwd, al64);
}

__global__ void __launch_bounds__(kMaxTileThreads)
    k_bwd_s(const Desc* __restrict__ D, const uint2* __restrict__ ranges, const uint32_t* __restrict__ pv,
            const float4* __restrict__ rec, const float4* __restrict__ box, float* __restrict__ g13,
            const uint32_t* __restrict__ order, Status* __restrict__ st, int persistent) {
  __shared__ WarpRecs s_w[kMaxTileThreads / 32];
  __shared__ uint32_t s_item[kMaxTileThreads / 32][32];
  const int lane = threadIdx.x & 31;
  WarpRecs& sw = s_w[threadIdx.x >> 5];
  uint32_t* si = s_item[threadIdx.x >> 5];
  uint32_t tile;
  uint32_t evals = 0, contrib = 0;
  for (int iter = 0; next_tile(persistent, order, D->n_tiles, &st->work_counter2, tile, iter); ++iter) {
    const TileCtx tc = tile_ctx(*D, tile, ranges, static_cast<int>(threadIdx.x));
    if (tc.end - tc.start > kLongList) continue;   // the long-list kernels' tile
    const FrameDev& F = D->f[tc.f];
    const WarpBox wb = warp_box(tc.inside, tc.r, tc.c, F.W);
    float dx = 0.f, dy = 0.f, dz = 0.f;
    float T = 1.f, gA = 0.f, gSt = 0.f, gSx = 0.f, gSy = 0.f, gSz = 0.f;
    int nc = 0;
    if (tc.inside) {
      pixel_ray(F, tc.r, tc.c, dx, dy, dz);
      T = F.Tf[tc.pix];
      nc = F.nc[tc.pix];
      gA = F.gA[tc.pix];
      gSt = F.gSt[tc.pix];
      gSx = F.gSn[tc.pix];
      gSy = F.gSn[tc.HW + tc.pix];
      gSz = F.gSn[2 * static_cast<int64_t>(tc.HW) + tc.pix];
    }
    // n_contrib comes from the caller: never walk past the tile's list
    const uint32_t len = tc.end - tc.start;
    const uint32_t stop = min(static_cast<uint32_t>(__reduce_max_sync(0xffffffffu, nc > 0 ? nc : 0)), len);
    float S = 0.f;
    for (int c0 = static_cast<int>((stop + 31) / 32) - 1; c0 >= 0; --c0) {
      const int k0 = 32 * c0;
      uint32_t item = 0;
      bool hit = false;
      if (static_cast<uint32_t>(k0 + lane) < stop) {
        item = __ldg(pv + tc.start + k0 + lane);
        hit = box_hits(__ldg(box + item), wb);
      }
      uint32_t m = __ballot_sync(0xffffffffu, hit);
      if (!m) continue;
      __syncwarp();
      if (hit) {
        stage_hit(rec, item, sw, lane);
        si[lane] = item;
      }
      __syncwarp();
      do {
        const int bq = 31 - __clz(m);
        m &= ~(1u << bq);
        const bool in = k0 + bq < nc;
        const float4 r0 = sw.r0[bq];
        Eval e;
        eval_pair(r0, sw.r1[bq], sw.r2[bq], sw.al[bq], dx, dy, dz, e);
        const bool valid = in && e.valid;
        evals += in;
        contrib += valid;
        if (!__any_sync(0xffffffffu, valid)) continue;
        // invalid lanes: zero opacity and finite inputs, so every moment is
        // exactly 0 and T, S pass through unchanged
        const float a = valid ? e.a : 0.f;
        const float araw = valid ? e.araw : 0.f;
        const float t = valid ? e.t : 0.f;
        const float u = valid ? e.u : 0.f;
        const float v = valid ? e.v : 0.f;
        const float rden = valid ? e.rden : 0.f;
        const float iom = rcp_ftz(1.0f - a);
        const float Tk = T * iom;
        const float sg = e.den > 0.f ? -1.f : 1.f;
        const float gc = gA + gSt * t + sg * (gSx * r0.x + gSy * r0.y + gSz * r0.z);
        const float w = a * Tk;
        const float dLda = Tk * gc - S * iom;
        S = fmaf(w, gc, S);
        T = Tk;
        const float g = araw < 0.99f ? araw * dLda : 0.f;
        const float ug = u * g, vg = v * g;
        const float ct = fmaf(w, gSt, -fmaf(ug, e.ud, vg * e.vd)) * rden;
        const float wsg = w * sg;
        float mv[12];
        mv[0] = g;
        mv[1] = ug;
        mv[2] = vg;
        mv[3] = u * ug;
        mv[4] = v * vg;
        mv[5] = u * vg;
        mv[6] = ct;
        mv[7] = ct * u;
        mv[8] = ct * v;
        mv[9] = wsg * gSx;
        mv[10] = wsg * gSy;
        mv[11] = wsg * gSz;
        int idx;
        const float r = warp_reduce12(mv, lane, idx);
        if (idx >= 0 && r != 0.f) atomicAdd(g13 + 16 * static_cast<int64_t>(si[bq]) + idx, r);
      } while (m);
    }
  }
  unsigned long long ev = evals, co = contrib;
  for (int o = 16; o > 0; o >>= 1) {
    ev += __shfl_xor_sync(0xffffffffu, ev, o);
    co += __shfl_xor_sync(0xffffffffu, co, o);
  }
  if (lane == 0 && ev) atomicAdd(&st->evals_bwd, ev);
  if (lane == 0 && co) atomicAdd(&st->contrib_bwd, co);
}

// ---------------------------------------------------------------------------
// Chunked backward (group 16 after the shared-memory forward): a work item
// is one warp's 4 x 8 pixel block of a tile over one chunk of kChunk list
// entries, claimed through an atomic counter from k_bwd_prep's queues: only
// chunks that hold one of the block's composited entries, chunks walked in
// full first, then the last ones by decreasing walked length (a warp that
// claims late gets a short item, so the SMs finish together).  The reverse
// walk of chunk c starts from the forward's checkpoint: T at the end of the
// chunk, and the suffix S = sum over the later chunks c' of gA dA_c' + gSt
// dSt_c' + gS . dSn_c' (their own sums of w, w t, w n').  Items are
// independent, so a frame offers several times more warps than pixel
// blocks.
// ---------------------------------------------------------------------------
constexpr int kBwdChunkCta = 128;

// A hit's 12 moments are summed over its pixels in two phases.  Phase A walks
// the chunk's hits one by one, as every lane's recurrence of T and S needs; a
// lane whose pixel composited the hit leaves its contribution (g, u, v, ct;
// w sg gS) in the warp's next free slots of shared memory.  Phase B, once
// kBwdHits hits are waiting or the slots are full, sums them with four lanes
// per hit and adds the moments with three 16-byte reductions, once per hit:
// of one hit the sum is always the same, only the hits' order varies.
// Contributions wait across chunks and tiles: the sums need nothing of where
// they came from but the item.
//
// Bound by issue (74 % of the cycles) and the latency of the chunk's six
// dependent reads.  Before, the 12 moments were summed over the warp with
// shuffles hit by hit and added by 12 lanes with scalar atomics: 162
// instructions a hit on the street frame (200k surfels, 128 x 1024), of whose
// 32 lanes 8 held a contribution; now 125.  Kernel 131 -> 113 us, its step 335 ->
// 318 us; the steps of 8 keyframes of a dense 1M map (12 lanes of 32) and of six
// batched maps gain 0.4 and 0.5 %.  Slots, the three steps: 96 318, 5728 and
// 4226 us; 128 317, 5710 and 4260; 80 324, 5750 and 4244
// (more shared memory leaves less L1 to the batched maps' reads).  Others: one
// lane per 4 contributions, each with its own three reductions, 313 and 5690 us,
// but twice the additions in an order that varies (results of two runs differed
// more than before); the same with the hit's lanes added up first 328 and 5760;
// every lane walking its own pixel's bits 322 and 6085 before the binning's last
// change (its record reads from shared memory conflict); two hits' evaluations
// at a time 330 and 6340 (128 registers); the next chunk claimed ahead 346 (a
// street frame has four chunks per warp: the last ones no longer balance).
constexpr int kBwdHits = 8;          // hits summed at a time
constexpr uint32_t kBwdSlots = 96;   // at least a hit's 32

struct BwdWarp {
  WarpRecs rec;
  float4 a[kBwdSlots];   // (g, u, v, ct)
  float4 b[kBwdSlots];   // (w sg gS, 0)
  uint32_t item[32];     // items of the staged hits
  uint32_t who[kChunk];  // the chunk's hits, last first: the pixels that composited them
  uint8_t entry[kChunk]; // and their entries of the chunk
};

// 16-byte aligned vector reduction into global memory.
__device__ __forceinline__ void red_add4(float* p, float x, float y, float z, float w) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

// Phase B: hit i < kBwdHits waits in the slots from lane i's `start` to lane
// i + 1's (`start` is the end for lanes past the last hit); `item` is its item.
__device__ __forceinline__ void bwd_flush(const BwdWarp& sb, uint32_t start, uint32_t item, float* __restrict__ g13,
                                          int lane) {
  static_assert(kBwdHits == 8, "four lanes per hit");
  __syncwarp();
  const uint32_t s0 = __shfl_sync(0xffffffffu, start, lane >> 2);
  const uint32_t s1 = __shfl_sync(0xffffffffu, start, (lane >> 2) + 1);
  const uint32_t it = __shfl_sync(0xffffffffu, item, lane >> 2);
  float v[12];
#pragma unroll
  for (int q = 0; q < 12; ++q) v[q] = 0.f;
  for (uint32_t i = s0 + (lane & 3); i < s1; i += 4) {
    const float4 a = sb.a[i], b = sb.b[i];
    const float ug = a.y * a.x, vg = a.z * a.x;
    v[0] += a.x;
    v[1] += ug;
    v[2] += vg;
    v[3] = fmaf(a.y, ug, v[3]);
    v[4] = fmaf(a.z, vg, v[4]);
    v[5] = fmaf(a.y, vg, v[5]);
    v[6] += a.w;
    v[7] = fmaf(a.w, a.y, v[7]);
    v[8] = fmaf(a.w, a.z, v[8]);
    v[9] += b.x;
    v[10] += b.y;
    v[11] += b.z;
  }
  // over the four lanes: lanes 0 and 1 of the four end with moments 0-3 and
  // 4-7, lane 2 with 8-11
  const bool up = lane & 2, odd = lane & 1;
  float k[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float hi = q < 4 ? v[8 + (q & 3)] : 0.f;
    k[q] = (up ? hi : v[q]) + __shfl_xor_sync(0xffffffffu, up ? v[q] : hi, 2);
  }
  float r[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    r[q] = (odd ? k[4 + q] : k[q]) + __shfl_xor_sync(0xffffffffu, odd ? k[q] : k[4 + q], 1);
  if (s1 > s0 && (lane & 3) < 3)
    red_add4(g13 + 16 * static_cast<int64_t>(it) + 4 * (lane & 3), r[0], r[1], r[2], r[3]);
  __syncwarp();
}

__global__ void __launch_bounds__(kBwdChunkCta, 7)
    k_bwd_c(const Desc* __restrict__ D, const uint2* __restrict__ ranges, const uint32_t* __restrict__ pv,
            const float4* __restrict__ rec, const float4* __restrict__ box, float* __restrict__ g13,
            const uint32_t* __restrict__ cbase, const float* __restrict__ ckpt, const uint32_t* __restrict__ cmask,
            SegBuf seg, const float* __restrict__ ssuf, const uint2* __restrict__ bq, uint32_t bq_cap0,
            uint32_t bq_capk, Status* __restrict__ st) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  __shared__ BwdWarp s_w[kBwdChunkCta / 32];
  const int lane = threadIdx.x & 31;
  BwdWarp& sb = s_w[threadIdx.x >> 5];
  WarpRecs& sw = sb.rec;
  uint32_t* si = sb.item;
  // the hits that wait for phase B: their count and slots (warp-uniform); lane i holds hit i's
  int waiting = 0;
  uint32_t used = 0, w_start = 0, w_item = 0;
  const int npx = D->th * D->tw, wpt = npx >> 5;
  // the forward's queues, claimed in class order: lane l < kBwdClasses holds
  // class l's size (clamped to its capacity) and the items before its end
  const uint32_t qn = lane < kBwdClasses ? min(st->bq_count[lane], lane == 0 ? bq_cap0 : bq_capk) : 0u;
  uint32_t qend = qn;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, qend, o);
    if (lane >= o) qend += x;
  }
  const uint32_t n_work = __shfl_sync(0xffffffffu, qend, kBwdClasses - 1);
  while (true) {
    uint32_t id = 0;
    if (lane == 0) id = atomicAdd(&st->work_counter2, 1u);
    id = __shfl_sync(0xffffffffu, id, 0);
    if (id >= n_work) break;
    const int cls = __ffs(__ballot_sync(0xffffffffu, lane < kBwdClasses && id < qend)) - 1;
    const uint32_t first = __shfl_sync(0xffffffffu, qend - qn, cls);
    const uint2 q = __ldg(bq + (cls == 0 ? 0u : bq_cap0 + static_cast<uint32_t>(cls - 1) * bq_capk) + (id - first));
    const uint32_t k = q.x / static_cast<uint32_t>(wpt);
    const int vt = static_cast<int>(q.x - k * static_cast<uint32_t>(wpt)) * 32 + lane;   // thread of the tile
    const uint32_t tile = q.y, c = k - __ldg(cbase + tile);
    const int f = frame_of_tile(*D, tile);
    const FrameDev& F = D->f[f];
    const int lt = static_cast<int>(tile - F.tile_base);
    const int ti = lt / F.ntc, tj = lt - ti * F.ntc;
    int lr, lc;
    pixel_of_thread(F, vt, lr, lc);
    const int r = ti * F.th + lr, col = tj * F.tw + lc;
    const bool inside = r < F.H && col < F.W;
    const int HW = F.H * F.W;
    const int64_t pix = static_cast<int64_t>(r) * F.W + col;
    const uint2 rg = ranges[tile];
    const int k_lo = static_cast<int>(c * kChunk);
    // n_contrib comes from the caller: never walk past the tile's list (its
    // chunks, segments and window masks end there)
    const int nc = inside ? min(F.nc[pix], static_cast<int>(rg.y - rg.x)) : 0;
    const bool act = nc > k_lo;
    float dx = 0.f, dy = 0.f, dz = 0.f;
    float T = 1.f, S = 0.f, gA = 0.f, gSt = 0.f, gSx = 0.f, gSy = 0.f, gSz = 0.f;
    if (act) {
      pixel_ray(F, r, col, dx, dy, dz);
      gA = F.gA[pix];
      gSt = F.gSt[pix];
      gSx = F.gSn[pix];
      gSy = F.gSn[HW + pix];
      gSz = F.gSn[2 * static_cast<int64_t>(HW) + pix];
      const float* o = ckpt + (static_cast<int64_t>(cbase[tile] + c) * kCkptSlots) * npx + vt;
      T = o[0];
      uint32_t c_last = static_cast<uint32_t>(nc - 1) / kChunk;
      if (rg.y - rg.x > kLongList) {
        // a long list: the segments after the chunk's are in the suffix that
        // k_bwd_prep wrote
        S = ssuf[static_cast<int64_t>(__ldg(seg.sbase + tile) + c / kSegChunks) * npx + vt];
        c_last = min(c_last, c / kSegChunks * kSegChunks + kSegChunks - 1);
      }
      for (uint32_t c2 = c + 1; c2 <= c_last; ++c2) {
        const float* q = ckpt + (static_cast<int64_t>(cbase[tile] + c2) * kCkptSlots) * npx + vt;
        S += gA * q[npx] + gSt * q[2 * npx] + gSx * q[3 * npx] + gSy * q[4 * npx] + gSz * q[5 * npx];
      }
    }
    // entries [k_lo, k_hi) of the list: the chunk's hits are the entries some
    // pixel of the warp composited (the forward's window masks), listed last
    // first with the pixels that did; their records are staged 32 hits at a time
    const uint32_t len = rg.y - rg.x;
    const int k_hi = static_cast<int>(min(min(static_cast<uint32_t>(k_lo) + kChunk, len),
                                          static_cast<uint32_t>(__reduce_max_sync(0xffffffffu, act ? nc : 0))));
    constexpr int kWin = kChunk / 32;
    uint32_t word[kWin];
    const int64_t cm = (static_cast<int64_t>(cbase[tile]) * 4 + static_cast<uint32_t>(k_lo) / 32) * npx + vt;
#pragma unroll
    for (int q = 0; q < kWin; ++q) {
      // entries below the pixel's n_contrib only (a long list's pixels stop
      // on their own, so their words past it are not this step's)
      const int lim = nc - k_lo - 32 * q;
      word[q] = act && lim > 0 && k_lo + 32 * q < k_hi ? __ldg(cmask + cm + static_cast<int64_t>(q) * npx) : 0u;
      if (lim < 32) word[q] &= lim > 0 ? (1u << lim) - 1u : 0u;
    }
    uint32_t hits = 0;
    __syncwarp();   // (the item before no longer reads the list)
#pragma unroll
    for (int q = kWin - 1; q >= 0; --q) {
      const uint32_t m = __reduce_or_sync(0xffffffffu, word[q]);
      if (!m) continue;
      const uint32_t px = warp_transpose(word[q], lane);
      if ((m >> lane) & 1u) {
        const uint32_t at = hits + static_cast<uint32_t>(__popc((m >> lane) >> 1));
        sb.who[at] = px;
        sb.entry[at] = static_cast<uint8_t>(32 * q + lane);
      }
      hits += static_cast<uint32_t>(__popc(m));
    }
    for (uint32_t b = 0; b < hits; b += 32) {
      __syncwarp();
      uint32_t my_who = 0;
      if (b + lane < hits) {
        my_who = sb.who[b + lane];
        const uint32_t item = __ldg(pv + rg.x + k_lo + sb.entry[b + lane]);
        stage_hit(rec, item, sw, lane);
        si[lane] = item;
      }
      __syncwarp();
      const int cnt = static_cast<int>(min(32u, hits - b));
      for (int j = 0; j < cnt; ++j) {
        // the pixels that composited this entry: their evaluation (the
        // forward's, bit for bit) is valid
        const uint32_t who = __shfl_sync(0xffffffffu, my_who, j);
        const uint32_t n = static_cast<uint32_t>(__popc(who));
        if (waiting == kBwdHits || used + n > kBwdSlots) {
          bwd_flush(sb, lane < waiting ? w_start : used, w_item, g13, lane);
          waiting = 0;
          used = 0;
        }
        if (lane == waiting) {
          w_start = used;
          w_item = si[j];
        }
        ++waiting;
        if ((who >> lane) & 1u) {
          const float4 r0 = sw.r0[j];
          Eval e;
          eval_pair(r0, sw.r1[j], sw.r2[j], sw.al[j], dx, dy, dz, e);
          const float iom = rcp_ftz(1.0f - e.a);
          const float Tk = T * iom;
          const float sg = e.den > 0.f ? -1.f : 1.f;
          const float gc = gA + gSt * e.t + sg * (gSx * r0.x + gSy * r0.y + gSz * r0.z);
          const float w = e.a * Tk;
          const float dLda = Tk * gc - S * iom;
          S = fmaf(w, gc, S);
          T = Tk;
          const float g = e.araw < 0.99f ? e.araw * dLda : 0.f;
          const float ct = fmaf(w, gSt, -fmaf(e.u * g, e.ud, e.v * g * e.vd)) * e.rden;
          const float wsg = w * sg;
          const uint32_t slot = used + static_cast<uint32_t>(__popc(who & ((1u << lane) - 1u)));
          sb.a[slot] = make_float4(g, e.u, e.v, ct);
          sb.b[slot] = make_float4(wsg * gSx, wsg * gSy, wsg * gSz, 0.f);
        }
        used += n;
      }
    }
  }
  if (waiting) bwd_flush(sb, lane < waiting ? w_start : used, w_item, g13, lane);
  // (the claim counter and the queue sizes are zeroed for the next backward by
  // k_preprocess_bwd, which follows on the stream; no statistics counters: the
  // backward's contributions are the forward's composited pairs, counted there)
}

// Long lists in the backward of the tunings without chunks: a work item is one
// (long tile, pixel), claimed through an atomic counter; the 32 lanes take 32
// consecutive entries of the list for the warp's pixel.  From T_final, the
// transmittance before each entry is T divided by the suffix product of (1 - a)
// over the lanes, the suffix S a suffix sum; every valid lane adds its own
// entry's 12 moments with atomics.
__global__ void __launch_bounds__(256) k_bwd_long(const Desc* __restrict__ D, const uint2* __restrict__ ranges,
                                                  const uint32_t* __restrict__ pv, const float4* __restrict__ rec,
                                                  const float4* __restrict__ box, float* __restrict__ g13,
                                                  const uint32_t* __restrict__ longt, Status* __restrict__ st) {
  const int lane = threadIdx.x & 31;
  const uint32_t n_long = st->n_long;
  if (n_long == 0) return;
  uint32_t evals = 0, contrib = 0;
  LongPix P;
  while (long_item(*D, ranges, longt, n_long, warp_claim(&st->long_counter_bwd), P)) {
    if (!P.inside) continue;
    const FrameDev& F = *P.F;
    const int nc = F.nc[P.pix];
    // n_contrib comes from the caller: never walk past the tile's list
    const uint32_t stop = min(static_cast<uint32_t>(nc > 0 ? nc : 0), P.end - P.start);
    if (stop == 0) continue;
    float dx, dy, dz;
    pixel_ray(F, P.r, P.c, dx, dy, dz);
    const float gA = F.gA[P.pix], gSt = F.gSt[P.pix];
    const float gSx = F.gSn[P.pix], gSy = F.gSn[P.HW + P.pix], gSz = F.gSn[2 * static_cast<int64_t>(P.HW) + P.pix];
    WarpBox pb;
    pb.r0 = pb.r1 = static_cast<float>(P.r);
    pb.cmid = static_cast<float>(P.c);
    pb.chalf = 0.f;
    pb.W = static_cast<float>(F.W);
    float T = F.Tf[P.pix], S = 0.f;
    for (int c0 = static_cast<int>((stop + 31) / 32) - 1; c0 >= 0; --c0) {
      const uint32_t k = 32u * c0 + lane;
      bool valid = false;
      Eval e;
      float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f);
      uint32_t item = 0;
      if (k < stop) {
        item = __ldg(pv + P.start + k);
        if (box_hits(__ldg(box + item), pb)) {
          const float4* rp = rec + 4 * static_cast<int64_t>(item);
          r0 = __ldg(rp);
          eval_pair(r0, __ldg(rp + 1), __ldg(rp + 2), __ldg(reinterpret_cast<const float*>(rp + 3)), dx, dy, dz, e);
          valid = e.valid;
          ++evals;
        }
      }
      const float om = valid ? 1.0f - e.a : 1.0f;
      // Q_j = prod_{i >= j} (1 - a_i) over the chunk's valid lanes
      float Qj = om;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_down_sync(0xffffffffu, Qj, o);
        if (lane + o < 32) Qj *= y;
      }
      const float Tk = __fdividef(T, Qj);   // transmittance before entry j
      float c = 0.f, gc = 0.f;
      if (valid) {
        const float sg = e.den > 0.f ? -1.f : 1.f;
        gc = gA + gSt * e.t + sg * (gSx * r0.x + gSy * r0.y + gSz * r0.z);
        c = e.a * Tk * gc;
      }
      // suffix sums of w (g.c): after entry j (exclusive) and over the chunk
      float Cs = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float y = __shfl_down_sync(0xffffffffu, Cs, o);
        if (lane + o < 32) Cs += y;
      }
      float Cex = __shfl_down_sync(0xffffffffu, Cs, 1);
      if (lane == 31) Cex = 0.f;
      if (valid) {
        ++contrib;
        float v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = 0.f;
        moments(e, r0, Tk, S + Cex, rcp_ftz(om), gA, gSt, gSx, gSy, gSz, v);
        float* gp = g13 + 16 * static_cast<int64_t>(item);
#pragma unroll
        for (int q = 0; q < kGrad; ++q)
          if (v[q] != 0.f) atomicAdd(gp + q, v[q]);
      }
      T = __fdividef(T, __shfl_sync(0xffffffffu, Qj, 0));
      S += __shfl_sync(0xffffffffu, Cs, 0);
    }
  }
  long_finish(&st->long_counter_bwd, &st->long_done_bwd, gridDim.x * (blockDim.x >> 5));
  unsigned long long ev = evals, co = contrib;
  for (int o = 16; o > 0; o >>= 1) {
    ev += __shfl_xor_sync(0xffffffffu, ev, o);
    co += __shfl_xor_sync(0xffffffffu, co, o);
  }
  if (lane == 0 && ev) atomicAdd(&st->evals_bwd, ev);
  if (lane == 0 && co) atomicAdd(&st->contrib_bwd, co);
}

// Before the chunked backward (one launch):
// (1) its work queues, from the forward's largest n_contrib of every (tile,
//     warp block): one thread per tile, warp-
//     aggregated reservations (one atomic per warp for class 0, one per
//     class present and block for the others).  A tile's full chunks are
//     queued chunk by chunk, its blocks side by side: they read the same
//     list entries, so warps that claim them together share those loads in
//     L2.  The queue sizes are zero on entry (cleared with the claim
//     counter).
// (2) over the long lists: the suffix S of every segment (the sum over the
//     pixel's later segments s' of gA dA_s' + gSt dSt_s' + gS . dSn_s'), so
//     that k_bwd_c sums the later chunks of one segment only instead of, per
//     work item, up to thousands of them.  One CTA per (long tile, warp
//     block): its eight warps split the block's segments into parts (lane =
//     pixel), sum their part while parking every segment's term in the suffix
//     buffer, add up the later parts' sums in shared memory, then walk their
//     part down.
constexpr int kMaxBlocks = kMaxTileThreads / 32;
constexpr uint32_t kPrepChunks = 16;   // full chunks that one lane queues

__global__ void __launch_bounds__(256) k_bwd_prep(const Desc* __restrict__ D, const uint2* __restrict__ ranges,
                                                  Status* __restrict__ st,
                                                  const uint32_t* __restrict__ cbase,
                                                  const uint32_t* __restrict__ bwm, uint2* __restrict__ bq,
                                                  uint32_t cap0, uint32_t capk, SegBuf seg,
                                                  float* __restrict__ ssuf) {
  pdl_wait();               // (launched after a kernel of this chain: wait for it)
  pdl_launch_dependents();  // the next kernel may be dispatched now
  const int lane = threadIdx.x & 31;
  const uint32_t blocks = static_cast<uint32_t>(D->th * D->tw) >> 5;
  const uint32_t n_tiles = D->n_tiles;
  // (1) a warp-uniform loop: every lane reaches the warp collectives
  for (uint32_t t0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); t0 < n_tiles; t0 += gridDim.x * blockDim.x) {
    const uint32_t tile = t0 + static_cast<uint32_t>(lane);
    const bool ok = tile < n_tiles;
    // (no word exceeds the list: a queued chunk is always one of the tile's)
    const uint2 rg = ok ? ranges[tile] : make_uint2(0u, 0u);
    uint32_t wm[kMaxBlocks];
    uint32_t nfull = 0, nf_max = 0;
#pragma unroll
    for (int b = 0; b < kMaxBlocks; ++b) {
      wm[b] = ok && static_cast<uint32_t>(b) < blocks ? min(bwm[tile * blocks + b], rg.y - rg.x) : 0u;
      nfull += wm[b] / kChunk;
      nf_max = max(nf_max, wm[b] / kChunk);
    }
    const uint32_t c0 = ok ? cbase[tile] : 0u;
    // class 0: the tile's full chunks, placed by an inclusive warp scan
    uint32_t incl = nfull;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    uint32_t pos = 0;
    if (lane == 31 && incl) pos = atomicAdd(&st->bq_count[0], incl);
    pos = __shfl_sync(0xffffffffu, pos, 31) + incl - nfull;
    // (a tile with more than a few full chunks is queued by the whole warp:
    // one lane writing a long list's thousands of items took 0.4 ms)
    const bool many = nf_max > kPrepChunks;
    for (uint32_t c = 0; c < (many ? 0u : nf_max); ++c) {
#pragma unroll
      for (int b = 0; b < kMaxBlocks; ++b) {
        if (c < wm[b] / kChunk) {
          if (pos < cap0) bq[pos] = make_uint2((c0 + c) * blocks + static_cast<uint32_t>(b), tile);
          ++pos;
        }
      }
    }
    for (uint32_t big = __ballot_sync(0xffffffffu, many); big; big &= big - 1) {
      const int src = __ffs(big) - 1;
      uint32_t full[kMaxBlocks];
#pragma unroll
      for (int b = 0; b < kMaxBlocks; ++b) full[b] = __shfl_sync(0xffffffffu, wm[b] / kChunk, src);
      const uint32_t nc = __shfl_sync(0xffffffffu, nf_max, src), cb = __shfl_sync(0xffffffffu, c0, src);
      uint32_t at = __shfl_sync(0xffffffffu, pos, src);
      for (uint32_t cc = 0; cc < nc; cc += 32) {
        const uint32_t c = cc + static_cast<uint32_t>(lane);
        uint32_t n = 0;
#pragma unroll
        for (int b = 0; b < kMaxBlocks; ++b) n += c < full[b];
        uint32_t o = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t x = __shfl_up_sync(0xffffffffu, o, d);
          if (lane >= d) o += x;
        }
        uint32_t k = at + o - n;
#pragma unroll
        for (int b = 0; b < kMaxBlocks; ++b)
          if (c < full[b]) {
            if (k < cap0) bq[k] = make_uint2((cb + c) * blocks + static_cast<uint32_t>(b), t0 + static_cast<uint32_t>(src));
            ++k;
          }
        at += __shfl_sync(0xffffffffu, o, 31);
      }
    }
    // every block's chunk holding its last entry: the class of its walked
    // length (longest first), one reservation per class present
#pragma unroll
    for (int b = 0; b < kMaxBlocks; ++b) {
      if (static_cast<uint32_t>(b) >= blocks) break;
      const uint32_t rem = wm[b] % kChunk;
      const uint32_t cls = rem ? 1u + ((kChunk - rem) * (kBwdClasses - 1)) / kChunk : 0u;
      const uint32_t peers = __match_any_sync(0xffffffffu, cls);
      const int leader = __ffs(peers) - 1;
      uint32_t bk = 0;
      if (cls && lane == leader) bk = atomicAdd(&st->bq_count[cls], static_cast<uint32_t>(__popc(peers)));
      bk = __shfl_sync(0xffffffffu, bk, leader) + static_cast<uint32_t>(__popc(peers & ((1u << lane) - 1u)));
      if (cls && bk < capk)
        bq[cap0 + (cls - 1) * capk + bk] = make_uint2((c0 + wm[b] / kChunk) * blocks + static_cast<uint32_t>(b), tile);
    }
  }
  // (2) requires 256 threads (eight parts); CTA-uniform loop
  __shared__ float s_part[8][32];
  const uint32_t n_long = st->n_long;
  const int npx = static_cast<int>(blocks) * 32;
  const int part = threadIdx.x >> 5;
  for (uint32_t it = blockIdx.x; it < n_long * blocks; it += gridDim.x) {
    const uint32_t lt = it / blocks, blk = it - lt * blocks;
    const uint32_t tile = seg.longt[lt];
    const int vt = static_cast<int>(blk) * 32 + lane;
    const TileCtx tc = tile_ctx(*D, tile, ranges, vt);
    const FrameDev& F = D->f[tc.f];
    // (the caller's n_contrib, at most the list)
    const int nc = tc.inside ? min(F.nc[tc.pix], static_cast<int>(tc.end - tc.start)) : 0;
    const int ns = nc > 0 ? (nc - 1) / static_cast<int>(kSeg) + 1 : 0;   // the pixel's segments
    const int per = (__reduce_max_sync(0xffffffffu, ns) + 7) / 8;
    const int lo = part * per, hi = min(lo + per, ns);
    float gA = 0.f, gSt = 0.f, gSx = 0.f, gSy = 0.f, gSz = 0.f;
    if (hi > lo) {
      gA = F.gA[tc.pix];
      gSt = F.gSt[tc.pix];
      gSx = F.gSn[tc.pix];
      gSy = F.gSn[tc.HW + tc.pix];
      gSz = F.gSn[2 * static_cast<int64_t>(tc.HW) + tc.pix];
    }
    const int64_t s0 = static_cast<int64_t>(seg.sbase[tile]);
    // pass 1: every segment's term (parked in ssuf) and the part's sum
    float tot = 0.f;
    for (int s = hi - 1; s >= lo; s -= 4) {
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[u] = 0.f;
        if (s - u >= lo) {
          const float* q = seg.sum + (s0 + s - u) * kSegSlots * npx + vt;
          v[u] = gA * q[0] + gSt * q[npx] + gSx * q[2 * npx] + gSy * q[3 * npx] + gSz * q[4 * npx];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (s - u >= lo) {
          ssuf[(s0 + s - u) * npx + vt] = v[u];
          tot += v[u];
        }
      }
    }
    s_part[part][lane] = tot;
    __syncthreads();
    float S = 0.f;
    for (int w2 = 7; w2 > part; --w2) S += s_part[w2][lane];
    // pass 2: the suffix after every segment of the part, walking down
    for (int s = hi - 1; s >= lo; s -= 8) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = s - u >= lo ? ssuf[(s0 + s - u) * npx + vt] : 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (s - u >= lo) {
          ssuf[(s0 + s - u) * npx + vt] = S;
          S += v[u];
        }
      }
    }
    __syncthreads();   // s_part is rewritten by the next item
  }
}

// The work counters start at zero (reset at binning and by the last warp of
// every launch), so no memset precedes the launch.
static cudaError_t launch_bwd_long(const WsPtrs& w, const uint32_t* pv, cudaStream_t s) {
  int dev = 0, sms = 152, per_sm = 2;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // as many CTAs as fit (the walks are bound by load latency); warps claim
  // (tile, pixel) items until none are left
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bwd_long, 256, 0);
  k_bwd_long<<<sms * (per_sm > 0 ? per_sm : 1), 256, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, w.g13, w.longt, w.st);
  return cudaGetLastError();
}

static SegBuf seg_buf(const WsPtrs& w) { return SegBuf{w.segs, w.longt, w.sbase, w.segsum, w.dead}; }

// Whether a map is large enough for a list to be long.
static bool may_be_long(const Desc& h) {
  int64_t most = 0;
  for (int f = 0; f < h.n_frames; ++f) most = h.f[f].n > most ? h.f[f].n : most;
  return most > static_cast<int64_t>(kLongList);
}

// 4 x 8 pixel blocks per warp (pixel_of_thread)
static bool block48(const Desc& h) { return (h.tw & 7) == 0 && (h.th & 3) == 0; }

// The long lists, before the tiles with short ones; `after_kernel`: they follow
// a kernel of this call.  Without long lists both are early exits whose launch
// overlaps the kernel before.
static cudaError_t launch_fwd_long(const WsPtrs& w, const Desc& h, const uint32_t* pv, cudaStream_t s,
                                   bool after_kernel, const LossEpi* loss) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const auto masks = block48(h) ? k_long_masks<true> : k_long_masks<false>;
  cudaError_t e;
  if (after_kernel) {
    e = launch_dep(masks, dim3(3 * sms), dim3(256), 0, s, w.desc, w.ranges, pv, w.rec, w.box, w.st, w.cbase, w.ckpt,
                   w.cmask, w.bwm, seg_buf(w));
  } else {
    masks<<<3 * sms, 256, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, w.st, w.cbase, w.ckpt, w.cmask, w.bwm,
                                  seg_buf(w));
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  return launch_dep(loss ? k_fwd_long<true> : k_fwd_long<false>, dim3(3 * sms), dim3(256), 0, s, w.desc, w.ranges, pv,
                    w.rec, w.st, w.cbase, w.ckpt, w.cmask, w.bwm, loss ? *loss : LossEpi{}, seg_buf(w));
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
template <int B>
static cudaError_t fwd_b(const WsPtrs& w, const uint32_t* pv, const Desc& h, int persistent, int grid, cudaStream_t s) {
  k_fwd<B><<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, persistent ? w.work : nullptr, w.st,
                                        persistent);
  return cudaGetLastError();
}

template <int B>
static cudaError_t bwd_b(const WsPtrs& w, const uint32_t* pv, const Desc& h, int persistent, int grid, cudaStream_t s) {
  k_bwd<B><<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, w.g13, persistent ? w.work : nullptr,
                                        w.st, persistent);
  return cudaGetLastError();
}

static int persistent_grid(int threads) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int per_sm = 2048 / (threads > 0 ? threads : 256);
  return sms * (per_sm < 1 ? 1 : per_sm);
}

// after_kernel: follows a kernel of this call
static cudaError_t launch_raster_fwd_tiles(const WsPtrs& w, const Desc& h, const uint32_t* pv, int batch,
                                           int group, int persistent, cudaStream_t s, bool after_kernel) {
  if (persistent) {
    cudaError_t e = cudaMemsetAsync(&w.st->work_counter, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
  }
  const int grid = persistent ? persistent_grid(h.th * h.tw) : static_cast<int>(h.n_tiles);
  const uint32_t* ord = persistent ? w.work : nullptr;
  switch (batch) {
    case 0:
      if (group == 16) {
        const auto fwd = block48(h) ? k_fwd_s<false, true> : k_fwd_s<false, false>;
        if (after_kernel && !persistent)   // (a persistent call's memset lies between)
          return launch_dep(fwd, dim3(grid), dim3(h.th * h.tw), 0, s, w.desc, w.ranges, pv, w.rec, w.box, ord, w.st,
                            persistent, w.cbase, w.ckpt, w.cmask, w.bwm, LossEpi{});
        fwd<<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, ord, w.st, persistent, w.cbase, w.ckpt,
                                         w.cmask, w.bwm, LossEpi{});
      } else if (group == 1) k_fwd_w<1><<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, ord, w.st, persistent);
      else if (group == 2) k_fwd_w<2><<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, ord, w.st, persistent);
      else k_fwd_w<4><<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, ord, w.st, persistent);
      return cudaGetLastError();
    case 64: return fwd_b<64>(w, pv, h, persistent, grid, s);
    case 128: return fwd_b<128>(w, pv, h, persistent, grid, s);
    case 512: return fwd_b<512>(w, pv, h, persistent, grid, s);
    default: return fwd_b<256>(w, pv, h, persistent, grid, s);
  }
}

static cudaError_t launch_raster_bwd_tiles(const WsPtrs& w, const Desc& h, const uint32_t* pv, int batch,
                                           int group, int persistent, cudaStream_t s) {
  if (persistent) {
    cudaError_t e = cudaMemsetAsync(&w.st->work_counter2, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
  }
  const int grid = persistent ? persistent_grid(h.th * h.tw) : static_cast<int>(h.n_tiles);
  const uint32_t* ord = persistent ? w.work : nullptr;
  switch (batch) {
    case 0:
      if (group == 16) k_bwd_s<<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, w.g13, ord, w.st, persistent);
      else if (group == 1) k_bwd_w<1><<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, w.g13, ord, w.st, persistent);
      else if (group == 2) k_bwd_w<2><<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, w.g13, ord, w.st, persistent);
      else k_bwd_w<4><<<grid, h.th * h.tw, 0, s>>>(w.desc, w.ranges, pv, w.rec, w.box, w.g13, ord, w.st, persistent);
      return cudaGetLastError();
    case 64: return bwd_b<64>(w, pv, h, persistent, grid, s);
    case 128: return bwd_b<128>(w, pv, h, persistent, grid, s);
    default: return bwd_b<256>(w, pv, h, persistent, grid, s);
  }
}

// The long lists, then the per-tile kernel, dispatched while they run (without long
// lists both are early exits; a plain launch waited for them: a render of 40,000
// surfels on a 128 x 2048 frame 113 us, now 108).
cudaError_t launch_raster_fwd(const Layout&, const WsPtrs& w, const Desc& h, const uint32_t* pv, int batch,
                              int group, int persistent, cudaStream_t s) {
  const bool longs = may_be_long(h);
  if (longs) {
    const cudaError_t e = launch_fwd_long(w, h, pv, s, false, nullptr);
    if (e != cudaSuccess) return e;
  }
  return launch_raster_fwd_tiles(w, h, pv, batch, group, persistent, s, longs);
}

int raster_fwd_kernel_count(const Desc& h) { return may_be_long(h) ? 3 : 1; }

// Chunked backward: as many resident CTAs as fit, warps claim (chunk, pixel
// block) items from the queues k_bwd_prep built until none are left.
static cudaError_t launch_raster_bwd_chunks(const WsPtrs& w, const uint32_t* pv, cudaStream_t s) {
  int dev = 0, sms = 152, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bwd_c, kBwdChunkCta, 0);
  return launch_dep(k_bwd_c, dim3(sms * (per_sm > 0 ? per_sm : 1)), dim3(kBwdChunkCta), 0, s, w.desc, w.ranges, pv,
                    w.rec, w.box, w.g13, w.cbase, w.ckpt, w.cmask, seg_buf(w), w.ssuf, w.bq, w.bq_cap0, w.bq_capk,
                    w.st);
}

// The shared-memory forward with the image-loss epilogue.  Follows
// launch_loss_counts on the same stream, which zeroed the tile counter.
cudaError_t launch_raster_fwd_loss(const WsPtrs& w, const Desc& h, const uint32_t* pv, int persistent,
                                   const lgs_loss_params& p, float* loss_out, cudaStream_t s) {
  LossEpi loss{p, loss_counts_ptr(w), reinterpret_cast<unsigned long long*>(w.loss_part), loss_out};
  const int grid = persistent ? persistent_grid(h.th * h.tw) : static_cast<int>(h.n_tiles);
  // (each follows a kernel of this call, k_loss_count first: dispatched while
  // it runs)
  if (may_be_long(h)) {
    const cudaError_t e = launch_fwd_long(w, h, pv, s, true, &loss);
    if (e != cudaSuccess) return e;
  }
  return launch_dep(block48(h) ? k_fwd_s<true, true> : k_fwd_s<true, false>, dim3(grid), dim3(h.th * h.tw), 0, s, w.desc,
                    w.ranges, pv, w.rec, w.box, persistent ? w.work : nullptr, w.st, persistent, w.cbase, w.ckpt,
                    w.cmask, w.bwm, loss);
}

cudaError_t launch_raster_bwd(const Layout&, const WsPtrs& w, const Desc& h, const uint32_t* pv, int batch,
                              int group, int persistent, bool chunked, cudaStream_t s) {
  if (chunked) {
    // the claim counter and the queue sizes are zero here (cleared at
    // binning and after every backward by k_preprocess_bwd); the queues and
    // the long lists' suffixes, then the walk
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    k_bwd_prep<<<4 * sms, 256, 0, s>>>(w.desc, w.ranges, w.st, w.cbase, w.bwm, w.bq, w.bq_cap0, w.bq_capk,
                                       seg_buf(w), w.ssuf);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_raster_bwd_chunks(w, pv, s);
  }
  cudaError_t e = launch_raster_bwd_tiles(w, h, pv, batch, group, persistent, s);
  if (e != cudaSuccess) return e;
  return launch_bwd_long(w, pv, s);
}

}  // namespace lgs
