// World radius of every point for stochastic point discarding (Sec. 3.1,
// "Stochastic Point Discarding": r_world = distance to the k-th nearest
// point, k = 4 in the paper), exact, on a hashed uniform grid.
//
//   1. bounding box (float min/max as ordered integers, atomics)
//   2. cell size h: 1.5 times the median k-NN distance of 256 sampled points,
//      exact (k_sample_bound, k_sample_scan, k_sample_select; the only host
//      synchronisation follows)
//   3. counting sort of the points by the hash of their search cell (1.6 h)
//   4. per point, in sorted order: the 8 search cells nearest to it (k_query);
//      points that these do not settle search a wider cube (k_query_far)
//   5. points whose search cells hold too many candidates: steps 3 and 4 again
//      for them alone, on cells of h / 8, nearest cells first (k_query_dense)
// 5M points on 50 surfaces: 8.73 ms with one block per sample and the points
// queried in input order cell by cell, 1.12 ms now.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <vector>

#include "launch.h"

namespace adop {
namespace knn {
namespace {

constexpr int kMaxK = 16;
constexpr int kSamples = 256;

__device__ __forceinline__ uint32_t ordered(float f) {
  const uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float unordered(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

__global__ void __launch_bounds__(256) k_bbox(const float* __restrict__ xyz, int64_t n, uint32_t* box) {
  uint32_t lo[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, hi[3] = {0u, 0u, 0u};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    for (int d = 0; d < 3; ++d) {
      const uint32_t o = ordered(__ldg(xyz + 3 * i + d));
      lo[d] = min(lo[d], o);
      hi[d] = max(hi[d], o);
    }
  // one atomic per block and bound: 58 thousand same-address atomics of a
  // warp each took 51 us on 5M points, whose 60 MB are a 9 us read
  __shared__ uint32_t s_lo[3][8], s_hi[3][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int d = 0; d < 3; ++d) {
    const uint32_t l = __reduce_min_sync(0xffffffffu, lo[d]), h = __reduce_max_sync(0xffffffffu, hi[d]);
    if (lane == 0) {
      s_lo[d][warp] = l;
      s_hi[d][warp] = h;
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    uint32_t l = 0xffffffffu, h = 0u;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) {
      l = min(l, s_lo[threadIdx.x][w]);
      h = max(h, s_hi[threadIdx.x][w]);
    }
    atomicMin(box + threadIdx.x, l);
    atomicMax(box + 3 + threadIdx.x, h);
  }
}

// The squared distance, one fixed sequence of operations: the sample kernels
// compare values that different kernels computed.
__device__ __forceinline__ float dist2(float dx, float dy, float dz) {
  return fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
}

// keep the k smallest values of a sorted ascending list
__device__ __forceinline__ void insert_k(float* best, int k, int& m, float d2) {
  if (m == k && d2 >= best[k - 1]) return;
  int q = m < k ? m++ : k - 1;
  while (q > 0 && best[q - 1] > d2) {
    best[q] = best[q - 1];
    --q;
  }
  best[q] = d2;
}

// The k-th smallest of a block's sorted lists (m entries in each thread), in
// thread 0; INFINITY if there are fewer.  k rounds of taking the least head,
// first in every warp, then over the warps' lists.
__device__ float block_kth(const float* best, int k, int m) {
  __shared__ float s_top[32][kMaxK];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  int at = 0;
  for (int r = 0; r < k; ++r) {  // (distances are >= 0: their bits order as they do)
    const uint32_t head = at < m ? __float_as_uint(best[at]) : 0x7f800000u;
    const uint32_t least = __reduce_min_sync(0xffffffffu, head);
    const unsigned who = __ballot_sync(0xffffffffu, head == least && at < m);
    if (who && lane == __ffs(who) - 1) ++at;
    if (lane == 0) s_top[warp][r] = __uint_as_float(least);
  }
  __syncthreads();
  float kth = INFINITY;
  if (warp == 0) {
    at = 0;
    for (int r = 0; r < k; ++r) {
      const bool more = lane < warps && at < k;
      const uint32_t head = more ? __float_as_uint(s_top[lane][at]) : 0x7f800000u;
      const uint32_t least = __reduce_min_sync(0xffffffffu, head);
      const unsigned who = __ballot_sync(0xffffffffu, head == least && more);
      if (who && lane == __ffs(who) - 1) ++at;
      kth = __uint_as_float(least);
    }
  }
  return kth;
}

__device__ __forceinline__ int64_t sample_index(int b, int64_t n) { return (int64_t)b * n / kSamples; }

// The k-NN distance of the samples without 256 scans of the cloud (one block
// per sample took 6.2 of 8.7 ms on 5M points: 1.3 G distances on 256 blocks,
// each thread with a list in local memory):
//   k_sample_bound   a bound per sample: the k-th smallest squared distance
//                    to a subset -- the 8 groups of 32 consecutive points
//                    around it and 1 / 128 of the cloud (at least 32768
//                    points) in evenly spread groups of 32; four groups a
//                    warp in flight (one at a time: 207 us on 5M points)
//   k_sample_scan    every point against every sample's bound; about 128 k
//                    points of a cloud in random order pass and are listed.
//                    1024 points of a block first test their bounding box
//                    against each bound: where neighbours in memory are
//                    neighbours in space nearly every (block, sample) is
//                    skipped, and a random order costs 7 instructions a pair.
//   k_sample_select  the k-th smallest of the list, or of the whole cloud
//                    where a list ran over
// The result is the exact k-th smallest squared distance in every case.
constexpr int kSubGroup = 32;
constexpr int kSubLeast = 32768;   // points
constexpr int kListCap = 4096;
constexpr int kBoundThreads = 512;

__global__ void __launch_bounds__(kBoundThreads) k_sample_bound(const float* __restrict__ xyz, int64_t n, int k, int64_t groups,
                                                      float* bound, uint32_t* list_count) {
  const int64_t si = sample_index(blockIdx.x, n);
  const float px = __ldg(xyz + 3 * si), py = __ldg(xyz + 3 * si + 1), pz = __ldg(xyz + 3 * si + 2);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t total = (n + kSubGroup - 1) / kSubGroup;   // groups of the cloud
  const int64_t near0 = max((int64_t)0, min(si / kSubGroup - 4, total - 8)), near1 = min(near0 + 8, total);
  float best[kMaxK];
  int m = 0;
  // groups <= total evenly spread ones, and [near0, near1); none twice
  constexpr int kWarps = kBoundThreads / 32;
  const int64_t near = near1 - near0;
  for (int64_t g0 = warp; g0 < groups + near; g0 += 4 * kWarps) {
    float d2[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t g = g0 + u * kWarps;
      const int64_t at = g < near ? near0 + g : (g - near) * total / groups;
      const int64_t j = at * kSubGroup + lane;
      const bool skip = g >= groups + near || (g >= near && at >= near0 && at < near1) || j >= n || j == si;
      d2[u] = skip ? INFINITY
                   : dist2(__ldg(xyz + 3 * j) - px, __ldg(xyz + 3 * j + 1) - py, __ldg(xyz + 3 * j + 2) - pz);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (d2[u] < INFINITY) insert_k(best, k, m, d2[u]);
  }
  __syncwarp();
  const float kth = block_kth(best, k, m);
  if (threadIdx.x == 0) {
    bound[blockIdx.x] = kth;
    list_count[blockIdx.x] = 0u;
  }
}

__global__ void __launch_bounds__(256) k_sample_scan(const float* __restrict__ xyz, int64_t n,
                                                     const float* __restrict__ bound, uint32_t* list_count,
                                                     float* list) {
  __shared__ float4 s_sample[kSamples];
  __shared__ int s_pick[kSamples];
  __shared__ float s_box[6][8];
  __shared__ int s_n;
  static_assert(kSamples == 256, "one thread per sample");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  {
    const int64_t si = sample_index(threadIdx.x, n);
    s_sample[threadIdx.x] =
        make_float4(__ldg(xyz + 3 * si), __ldg(xyz + 3 * si + 1), __ldg(xyz + 3 * si + 2), bound[threadIdx.x]);
  }
  for (int64_t t0 = (int64_t)blockIdx.x * 1024; t0 < n; t0 += (int64_t)gridDim.x * 1024) {
    float x[4], y[4], z[4];
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t j = t0 + u * 256 + threadIdx.x;
      const bool in = j < n;
      x[u] = in ? __ldg(xyz + 3 * j) : INFINITY;  // (an infinite distance passes no finite bound)
      y[u] = in ? __ldg(xyz + 3 * j + 1) : INFINITY;
      z[u] = in ? __ldg(xyz + 3 * j + 2) : INFINITY;
      if (in) {
        lo[0] = fminf(lo[0], x[u]); hi[0] = fmaxf(hi[0], x[u]);
        lo[1] = fminf(lo[1], y[u]); hi[1] = fmaxf(hi[1], y[u]);
        lo[2] = fminf(lo[2], z[u]); hi[2] = fmaxf(hi[2], z[u]);
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
        hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
      }
      if (lane == 0) {
        s_box[d][warp] = lo[d];
        s_box[3 + d][warp] = hi[d];
      }
    }
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    {  // thread t: can any point of the box be within sample t's bound?  (FP32
       // subtraction, max and dist2 are monotone, so no point that passes below is lost)
      const float4 q = s_sample[threadIdx.x];
      float bl[3], bh[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        bl[d] = s_box[d][0];
        bh[d] = s_box[3 + d][0];
#pragma unroll
        for (int w = 1; w < 8; ++w) {
          bl[d] = fminf(bl[d], s_box[d][w]);
          bh[d] = fmaxf(bh[d], s_box[3 + d][w]);
        }
      }
      const float dx = fmaxf(fmaxf(bl[0] - q.x, q.x - bh[0]), 0.0f);
      const float dy = fmaxf(fmaxf(bl[1] - q.y, q.y - bh[1]), 0.0f);
      const float dz = fmaxf(fmaxf(bl[2] - q.z, q.z - bh[2]), 0.0f);
      if (dist2(dx, dy, dz) <= q.w) s_pick[atomicAdd(&s_n, 1)] = threadIdx.x;
    }
    __syncthreads();
    const int picked = s_n;
    for (int r = 0; r < picked; ++r) {
      const int t = s_pick[r];
      const float4 q = s_sample[t];
      float d2[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) d2[u] = dist2(x[u] - q.x, y[u] - q.y, z[u] - q.z);
      if (!(fminf(fminf(d2[0], d2[1]), fminf(d2[2], d2[3])) <= q.w)) continue;
      const int64_t si = sample_index(t, n);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t j = t0 + u * 256 + threadIdx.x;
        if (d2[u] <= q.w && j < n && j != si) {
          const uint32_t slot = atomicAdd(list_count + t, 1u);
          if (slot < kListCap) list[(size_t)t * kListCap + slot] = d2[u];
        }
      }
    }
    __syncthreads();
  }
}

// out[s] = the k-NN distance of sample s.  scanned: whether k_sample_scan ran
// (else the bound came from the whole cloud).
__global__ void __launch_bounds__(256) k_sample_select(const float* __restrict__ xyz, int64_t n, int k, int scanned,
                                                       const float* __restrict__ bound,
                                                       const uint32_t* __restrict__ list_count,
                                                       const float* __restrict__ list, float* out) {
  float kth = bound[blockIdx.x];
  if (scanned) {
    const uint32_t count = list_count[blockIdx.x];
    float best[kMaxK];
    int m = 0;
    if (count <= kListCap) {
      for (uint32_t j = threadIdx.x; j < count; j += blockDim.x)
        insert_k(best, k, m, list[(size_t)blockIdx.x * kListCap + j]);
    } else {
      const int64_t si = sample_index(blockIdx.x, n);
      const float px = __ldg(xyz + 3 * si), py = __ldg(xyz + 3 * si + 1), pz = __ldg(xyz + 3 * si + 2);
      for (int64_t j = threadIdx.x; j < n; j += blockDim.x)
        if (j != si)
          insert_k(best, k, m, dist2(__ldg(xyz + 3 * j) - px, __ldg(xyz + 3 * j + 1) - py, __ldg(xyz + 3 * j + 2) - pz));
    }
    __syncwarp();
    kth = block_kth(best, k, m);
  }
  if (threadIdx.x == 0) out[blockIdx.x] = sqrtf(kth);
}

// Two grids over the bounding box: cells of h, which bound how far a search
// goes, and search cells of kSearch h, which hold the sorted points.
struct Grid {
  float ox, oy, oz;
  float inv_h, inv_s;  // 1 / h, 1 / (kSearch h)
  float s2_low;        // (kSearch h)^2, a little less: squared distances in search cells times this are lower bounds
  float slack;         // in search cells: the rounding of two points' cell coordinates
  uint32_t mask;       // buckets - 1
};

__device__ __forceinline__ void cell_of(const Grid& g, float inv, float x, float y, float z, int& cx, int& cy, int& cz) {
  cx = (int)floorf((x - g.ox) * inv);
  cy = (int)floorf((y - g.oy) * inv);
  cz = (int)floorf((z - g.oz) * inv);
}

// Bucket of a search cell: a multiplicative hash with the first rounds of
// murmur3's 32-bit finalizer, so that the few occupied cells of a surface
// spread over the table.
__device__ __forceinline__ uint32_t bucket(const Grid& g, int Cx, int Cy, int Cz) {
  uint32_t v = ((uint32_t)Cx * 73856093u) ^ ((uint32_t)Cy * 19349663u) ^ ((uint32_t)Cz * 83492791u);
  v ^= v >> 16;
  v *= 0x85ebca6bu;
  v ^= v >> 13;
  return v & g.mask;
}

// Tells apart the cells that share a bucket.  Two cells of one search (at most
// 14 apart along an axis) never have the same tag, so no point is met twice; a
// distant point with the same tag and bucket is met as the distant point that
// it is.
__device__ __forceinline__ uint32_t cell_tag(int Cx, int Cy, int Cz) {
  return (uint32_t)Cx + ((uint32_t)Cy << 10) + ((uint32_t)Cz << 20);
}

// Counts every bucket and keeps the count's old value, the point's rank in
// its bucket, so that the scatter needs no atomics.  Four points a thread, so
// that their round trips overlap.
constexpr int kAhead = 4;

// (The sort's steps read with plain loads what the step before wrote: they also
// run one after the other within k_query_dense.)
__device__ __forceinline__ void count_points(const float* xyz, int64_t n, const Grid& g, uint2* bkt, uint32_t* count) {
  const int64_t S = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += kAhead * S) {
    uint32_t b[kAhead], rank[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int64_t i = min(i0 + u * S, n - 1);
      int cx, cy, cz;
      cell_of(g, g.inv_s, __ldg(xyz + 3 * i), __ldg(xyz + 3 * i + 1), __ldg(xyz + 3 * i + 2), cx, cy, cz);
      b[u] = bucket(g, cx, cy, cz);
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (i0 + u * S < n) rank[u] = atomicAdd(count + b[u], 1u);
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (i0 + u * S < n) bkt[i0 + u * S] = make_uint2(b[u], rank[u]);
  }
}

__global__ void __launch_bounds__(256) k_count(const float* __restrict__ xyz, int64_t n, Grid g,
                                               uint2* __restrict__ bkt, uint32_t* __restrict__ count) {
  count_points(xyz, n, g, bkt, count);
}

// Exclusive scan of `count` (length m) into `start` (length m + 1), three
// phases over tiles of 4096 entries, by blocks of T threads.
constexpr int kScanTile = 4096;

// This thread's exclusive prefix of v over its block.
template <int T>
__device__ __forceinline__ uint32_t block_prefix(uint32_t v) {
  __shared__ uint32_t warp_sum[T / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < T / 32 ? warp_sum[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < T / 32) warp_sum[lane] = w;
  }
  __syncthreads();
  const uint32_t before = incl - v + (warp > 0 ? warp_sum[warp - 1] : 0u);
  __syncthreads();  // (the block may call again)
  return before;
}

template <int T>
__device__ __forceinline__ void scan_tile(const uint32_t* count, int64_t m, int64_t tile, uint32_t* tile_sum) {
  const int64_t t0 = tile * kScanTile + threadIdx.x * (kScanTile / T);
  uint32_t s = 0;
#pragma unroll
  for (int q = 0; q < kScanTile / T; ++q)
    if (t0 + q < m) s += count[t0 + q];
  const uint32_t before = block_prefix<T>(s);
  if (threadIdx.x == T - 1) tile_sum[tile] = before + s;
}

// one block: exclusive scan of the tile sums, serial chunks per thread
template <int T>
__device__ __forceinline__ void scan_sums(uint32_t* tile_sum, int64_t tiles) {
  const int64_t per = (tiles + T - 1) / T;
  const int64_t a = threadIdx.x * per, b = min(tiles, a + per);
  uint32_t local = 0;
  for (int64_t t = a; t < b; ++t) local += tile_sum[t];
  uint32_t run = block_prefix<T>(local);
  for (int64_t t = a; t < b; ++t) {
    const uint32_t v = tile_sum[t];
    tile_sum[t] = run;
    run += v;
  }
}

template <int T>
__device__ __forceinline__ void scan_apply(const uint32_t* count, int64_t m, int64_t tile, const uint32_t* tile_off,
                                           uint32_t* start, uint32_t total) {
  const int64_t t0 = tile * kScanTile + threadIdx.x * (kScanTile / T);
  uint32_t v[kScanTile / T], s = 0;
#pragma unroll
  for (int q = 0; q < kScanTile / T; ++q) {
    v[q] = t0 + q < m ? count[t0 + q] : 0u;
    s += v[q];
  }
  uint32_t run = tile_off[tile] + block_prefix<T>(s);
#pragma unroll
  for (int q = 0; q < kScanTile / T; ++q)
    if (t0 + q < m) {
      start[t0 + q] = run;
      run += v[q];
    }
  if (tile == 0 && threadIdx.x == 0) start[m] = total;
}

__global__ void __launch_bounds__(1024) k_scan_tiles(const uint32_t* __restrict__ count, int64_t m,
                                                     uint32_t* __restrict__ tile_sum) {
  scan_tile<1024>(count, m, blockIdx.x, tile_sum);
}

__global__ void __launch_bounds__(1024) k_scan_sums(uint32_t* __restrict__ tile_sum, int64_t tiles) {
  scan_sums<1024>(tile_sum, tiles);
}

__global__ void __launch_bounds__(1024) k_scan_apply(const uint32_t* __restrict__ count, int64_t m,
                                                     const uint32_t* __restrict__ tile_off, uint32_t* __restrict__ start,
                                                     uint32_t total) {
  scan_apply<1024>(count, m, blockIdx.x, tile_off, start, total);
}

__device__ __forceinline__ void scatter_points(const float* xyz, int64_t n, const Grid& g, const uint2* bkt,
                                               const uint32_t* start, float4* sorted, uint32_t* index) {
  const int64_t S = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += kAhead * S) {
    uint2 b[kAhead];
    float4 p[kAhead];
    uint32_t pos[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int64_t i = min(i0 + u * S, n - 1);
      b[u] = bkt[i];
      p[u].x = __ldg(xyz + 3 * i);
      p[u].y = __ldg(xyz + 3 * i + 1);
      p[u].z = __ldg(xyz + 3 * i + 2);
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) pos[u] = start[b[u].x] + b[u].y;
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      if (i0 + u * S >= n) continue;
      int cx, cy, cz;
      cell_of(g, g.inv_s, p[u].x, p[u].y, p[u].z, cx, cy, cz);
      p[u].w = __uint_as_float(cell_tag(cx, cy, cz));
      sorted[pos[u]] = p[u];
      index[pos[u]] = (uint32_t)(i0 + u * S);
    }
  }
}

__global__ void __launch_bounds__(256) k_scatter(const float* __restrict__ xyz, int64_t n, Grid g,
                                                 const uint2* __restrict__ bkt, const uint32_t* __restrict__ start,
                                                 float4* __restrict__ sorted, uint32_t* __restrict__ index) {
  scatter_points(xyz, n, g, bkt, start, sorted, index);
}

// The search is bounded: a point's result is the k-th smallest distance to
// the points at most kMaxRing cells away along each axis (+inf if there are
// fewer than k) -- the exact result unless the true neighbour is further than
// that, else an upper bound.  k_query looks at kMaxScan candidates at most and
// each lane of k_query_far at as many per ball; a point that has more is
// searched again by k_query_dense, on cells of h / kFine from the nearest
// outwards, and only there, after another kMaxScan candidates, does the
// smallest found so far stand (more points than that in cells of h / kFine, or
// of 2^-20 of the box where that is wider, around a point that are no copies
// of it).
constexpr int kMaxRing = 8;
constexpr int kMaxScan = 1 << 16;
constexpr float kFine = 8.0f;

// What is left: points listed for k_query_far, listed for k_query_dense, and
// passed on to it by k_query_far.
enum Counts { kListed = 0, kDense = 1, kMarked = 2 };

// The K smallest squared distances met, ascending; +inf where there are fewer.
template <int K>
struct Nearest {
  float d[K];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int q = 0; q < K; ++q) d[q] = INFINITY;
  }
  __device__ __forceinline__ void insert(float v) {  // v < d[K - 1]
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const float lo = fminf(d[q], v);
      v = fmaxf(d[q], v);
      d[q] = lo;
    }
  }
  // the k-th smallest, k <= K (K = 4 serves k = 4 alone, so that d stays in registers)
  __device__ __forceinline__ float kth(int k) const { return K == 4 ? d[3] : d[k - 1]; }
};

// One thread per point, in sorted order, so that the lanes of a warp look at
// the same buckets.  A point looks at the 2 x 2 x 2 search cells nearest to it:
// its own and the neighbours on the nearer side of each axis, so everything
// nearer than half a search cell, and up to a whole one, is among them.  The
// non-empty ranges go to shared memory first and the candidates of all of
// them form one loop: with a loop per cell a warp ran the longest range of its
// lanes eight times over (983 us on 5M points under ncu, 76% issue active; now
// 781 us).  Bound by instruction issue and, the candidates of a warp lying in
// several cells, by the L1: 32 KB of ranges a block instead of 16 cost it its
// L1 share and 1050 us, 40 registers (6 blocks per SM) 900 us.  Search cells of 1.6 h: 38
// candidates a point on a jittered surface; 2 h: 60, 1.25 h: 24 but 23% of the
// points unsettled.  The unsettled ones are listed for k_query_far with their
// distance so far in radius.  K = 4 (in registers) for k = 4, else 16.
constexpr float kSearch = 1.6f;

template <int K>
__global__ void __launch_bounds__(256) k_query(int64_t n, int k, Grid g, const uint32_t* __restrict__ start,
                                               const float4* __restrict__ sorted,
                                               const uint32_t* __restrict__ index, float* __restrict__ radius,
                                               uint32_t* __restrict__ pending, uint32_t* __restrict__ counts) {
  __shared__ uint2 s_range[8][256];  // first point, count and octant
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const float4 p = __ldg(sorted + i);
    int cx, cy, cz;
    cell_of(g, g.inv_s, p.x, p.y, p.z, cx, cy, cz);
    // per axis: the nearer neighbour, and the distance to it in search cells
    const float ux = (p.x - g.ox) * g.inv_s - (float)cx, uy = (p.y - g.oy) * g.inv_s - (float)cy,
                uz = (p.z - g.oz) * g.inv_s - (float)cz;
    const int sx = ux < 0.5f ? -1 : 1, sy = uy < 0.5f ? -1 : 1, sz = uz < 0.5f ? -1 : 1;
    const float near = fmaxf(fminf(ux, 1.0f - ux), fmaxf(fminf(uy, 1.0f - uy), fminf(uz, 1.0f - uz)));
    int ranges = 0, scanned = 0;
    uint32_t rs[8], re[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) {  // own cell first
      const uint32_t b = bucket(g, cx + ((o & 1) ? sx : 0), cy + ((o & 2) ? sy : 0), cz + ((o & 4) ? sz : 0));
      rs[o] = __ldg(start + b);
      re[o] = __ldg(start + b + 1);
    }
#pragma unroll
    for (int o = 0; o < 8; ++o) {
      const int len = (int)min(re[o] - rs[o], (uint32_t)(kMaxScan - scanned));
      if (len > 0)
        s_range[ranges++][threadIdx.x] = make_uint2(rs[o], (uint32_t)len | ((uint32_t)o << 20));
      scanned += len;
    }
    Nearest<K> best;
    best.clear();
    uint32_t s = 0, e = 0, tag = 0;
    const uint32_t own_tag = cell_tag(cx, cy, cz), tx = (uint32_t)sx, ty = (uint32_t)sy << 10, tz = (uint32_t)sz << 20;
    for (int r = 0;;) {
      if (s == e) {
        if (r == ranges || best.kth(k) == 0.0f) break;  // (k copies: nothing is closer)
        const uint2 v = s_range[r++][threadIdx.x];
        s = v.x;
        e = s + (v.y & 0xfffffu);
        tag = own_tag + ((v.y >> 20) & 1u) * tx + ((v.y >> 21) & 1u) * ty + (v.y >> 22) * tz;
      }
      const float4 q = __ldg(sorted + s);
      const float d2 = dist2(q.x - p.x, q.y - p.y, q.z - p.z);
      best.insert((__float_as_uint(q.w) == tag && s != (uint32_t)i) ? fminf(d2, INFINITY) : INFINITY);  // (NaN: no neighbour)
      ++s;
    }
    const float kth = best.kth(k);
    const float reach = fmaxf(1.0f - near - g.slack, 0.0f);
    const uint32_t at = __ldg(index + i);
    radius[at] = sqrtf(kth);
    // too many candidates: what was found is the best of a part of them.  These
    // points are listed from the end of `pending`, by their place in xyz
    if (scanned >= kMaxScan) {
      if (kth > 0.0f) pending[n - 1 - atomicAdd(counts + kDense, 1u)] = at;
    } else if (kth > reach * reach * g.s2_low) {
      pending[atomicAdd(counts + kListed, 1u)] = (uint32_t)i;
    }
  }
}

// The points that their nearest cells did not settle (1 in 100 of a jittered
// surface), a warp each, a cell a lane: the cells that a ball around the point
// meets, its radius the distance found so far (every nearer point is in it),
// or 4 h and 9 h (past which nothing counts) while fewer than k points were
// found.  (A thread each took 188 us on 5M points: few threads, each a chain
// of some 27 lookups.)  64 registers, 4 blocks per SM: with the 48 and 56 that
// the compiler settles on under other bounds the loop over a cell's points was
// slower (1M points of a curve 580 and 571 us, now 538).
constexpr uint32_t kMark = 0x80000000u;
constexpr int kDenseBlocksPerSm = 4;  // resident: 64 registers a thread

template <int K>
__global__ void __launch_bounds__(256, 4)
    k_query_far(int k, Grid g, const uint32_t* __restrict__ start, const float4* __restrict__ sorted,
                const uint32_t* __restrict__ index, int max_ring, float* __restrict__ radius,
                uint32_t* __restrict__ pending, uint32_t* __restrict__ counts) {
  const uint32_t count = counts[kListed];
  const int rings = min(max_ring, kMaxRing);
  const int lane = threadIdx.x & 31;
  const uint32_t warps = gridDim.x * (blockDim.x >> 5);
  for (uint32_t j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < count; j += warps) {  // warp-uniform
    const uint32_t i = pending[j];
    const float4 p = __ldg(sorted + i);
    const uint32_t at = __ldg(index + i);
    int cx, cy, cz;
    cell_of(g, g.inv_h, p.x, p.y, p.z, cx, cy, cz);
    const float fx = (p.x - g.ox) * g.inv_s, fy = (p.y - g.oy) * g.inv_s, fz = (p.z - g.oz) * g.inv_s;
    float found = radius[at];  // an upper bound of the result, or +inf
    const float most = (float)(rings + 1) / kSearch + g.slack;  // search cells that the cube of +-rings cells spans
    bool last, full;
    float ball = 0.0f;
    do {
      if (found < INFINITY) {
        ball = fminf(found * g.inv_s * 1.00001f + g.slack, most);
        last = true;
      } else {
        ball = ball == 0.0f ? fminf(4.0f / kSearch, most) : most;
        last = ball == most;
      }
      const float limit = found < INFINITY ? found * found * 1.00001f : INFINITY;
      Nearest<K> best;
      best.clear();
      int scanned = 0;
      const int x0 = (int)floorf(fx - ball), y0 = (int)floorf(fy - ball), z0 = (int)floorf(fz - ball);
      const int nx = (int)floorf(fx + ball) - x0 + 1, ny = (int)floorf(fy + ball) - y0 + 1,
                nz = (int)floorf(fz + ball) - z0 + 1;
      for (int c = lane; c < nx * ny * nz && scanned < kMaxScan; c += 32) {
        const int qx = x0 + c % nx, qy = y0 + c / nx % ny, qz = z0 + c / (nx * ny);
        const float dx = fmaxf(fmaxf((float)qx - fx, fx - (float)(qx + 1)) - g.slack, 0.0f);
        const float dy = fmaxf(fmaxf((float)qy - fy, fy - (float)(qy + 1)) - g.slack, 0.0f);
        const float dz = fmaxf(fmaxf((float)qz - fz, fz - (float)(qz + 1)) - g.slack, 0.0f);
        if ((dx * dx + dy * dy + dz * dz) * g.s2_low > limit) continue;
        const uint32_t b = bucket(g, qx, qy, qz), tag = cell_tag(qx, qy, qz);
        uint32_t s = __ldg(start + b);
        const uint32_t e = s + min(__ldg(start + b + 1) - s, (uint32_t)(kMaxScan - scanned));
        scanned += (int)(e - s);
        for (; s < e; ++s) {
          const float4 q = __ldg(sorted + s);
          const float d2 = dist2(q.x - p.x, q.y - p.y, q.z - p.z);
          if (!(d2 < best.d[K - 1]) || __float_as_uint(q.w) != tag || s == i) continue;
          int ox, oy, oz;  // the cube of +-rings cells bounds what counts
          cell_of(g, g.inv_h, q.x, q.y, q.z, ox, oy, oz);
          if (max(abs(ox - cx), max(abs(oy - cy), abs(oz - cz))) <= rings) best.insert(d2);
        }
      }
      __syncwarp();
      // the k-th smallest of the lanes' lists: k times the least head
      float kth = INFINITY;
      for (int r = 0; r < k; ++r) {  // (distances are >= 0: their bits order as they do)
        const uint32_t head = __float_as_uint(best.d[0]);
        const uint32_t least = __reduce_min_sync(0xffffffffu, head);
        const unsigned who = __ballot_sync(0xffffffffu, head == least);
        if (lane == __ffs(who) - 1) {
#pragma unroll
          for (int q = 0; q < K - 1; ++q) best.d[q] = best.d[q + 1];
          best.d[K - 1] = INFINITY;
        }
        kth = __uint_as_float(least);
      }
      found = sqrtf(kth);
      // the k-th of a first, smaller ball is exact if the ball reaches it
      if (found < INFINITY && found * g.inv_s * 1.00001f + g.slack <= ball) last = true;
      full = __any_sync(0xffffffffu, scanned >= kMaxScan);
    } while (!last && !full);
    if (lane == 0) {
      if (full) {  // (the point's place in xyz, marked: n < 2^31)
        found = fminf(found, radius[at]);
        pending[j] = at | kMark;
        atomicAdd(counts + kMarked, 1u);
      }
      radius[at] = found;
    }
  }
}

// The points with too many candidates, a warp each, over all points sorted
// again by cells of h / kFine: the cells around the point in shells, nearest
// first, a cell a lane to look up and the whole warp over each cell's points,
// until the k-th distance found is within the shells (or a shell is past what
// is known already: radius holds the best of the first search, or +inf).
// Sort and search are one cooperative launch, which ends at once (2.7 us) where
// there is no such point: six launches that end at once cost 27 us of a call on
// a thousand points (131 us), and asking on the host would be a second
// synchronisation.
template <int K>
__global__ void __launch_bounds__(256, kDenseBlocksPerSm)
    k_query_dense(const float* __restrict__ xyz, int64_t n, int k, Grid g, float most, uint2* bkt, uint32_t* count,
                  int64_t m, uint32_t* tiles, uint32_t* start, float4* sorted, uint32_t* index,
                  float* __restrict__ radius, const uint32_t* __restrict__ pending,
                  const uint32_t* __restrict__ counts) {
  if ((counts[kDense] | counts[kMarked]) == 0u) return;  // (every block alike)
  {
    const cooperative_groups::grid_group grid = cooperative_groups::this_grid();
    const int64_t nt = (m + kScanTile - 1) / kScanTile;
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < m; b += (int64_t)gridDim.x * blockDim.x) count[b] = 0u;
    grid.sync();
    count_points(xyz, n, g, bkt, count);
    grid.sync();
    for (int64_t t = blockIdx.x; t < nt; t += gridDim.x) scan_tile<256>(count, m, t, tiles);
    grid.sync();
    if (blockIdx.x == 0) scan_sums<256>(tiles, nt);
    grid.sync();
    for (int64_t t = blockIdx.x; t < nt; t += gridDim.x) scan_apply<256>(count, m, t, tiles, start, (uint32_t)n);
    grid.sync();
    scatter_points(xyz, n, g, bkt, start, sorted, index);
    grid.sync();
  }
  const uint32_t listed = counts[kListed], total = listed + counts[kDense];  // <= n < 2^31
  const int lane = threadIdx.x & 31;
  const uint32_t warps = gridDim.x * (blockDim.x >> 5);
  for (uint32_t j = (counts[kMarked] ? 0u : listed) + blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < total;
       j += warps) {  // warp-uniform
    const uint32_t entry = j < listed ? pending[j] : pending[n - 1 - (j - listed)] | kMark;
    if (!(entry & kMark)) continue;  // settled by k_query_far
    const int64_t at = entry & ~kMark;
    const float px = __ldg(xyz + 3 * at), py = __ldg(xyz + 3 * at + 1), pz = __ldg(xyz + 3 * at + 2);
    const uint2 own_slot = bkt[at];
    const uint32_t own = start[own_slot.x] + own_slot.y;
    int cx, cy, cz;
    cell_of(g, g.inv_s, px, py, pz, cx, cy, cz);
    const float fx = (px - g.ox) * g.inv_s, fy = (py - g.oy) * g.inv_s, fz = (pz - g.oz) * g.inv_s;
    const float known = radius[at];
    const float ball = known < INFINITY ? fminf(known * g.inv_s * 1.00001f + g.slack, most) : most;
    float limit = known < INFINITY ? known * known * 1.00001f : INFINITY;  // no further point counts
    float kth = INFINITY;
    int scanned = 0;
    Nearest<K> best;
    best.clear();
    for (int r = 0;; ++r) {
      const int side = 2 * r + 1, faces = 2 * side * side, layer = 8 * r;
      const int cells = r == 0 ? 1 : faces + (side - 2) * layer;
      for (int c0 = 0; c0 < cells && scanned < kMaxScan; c0 += 32) {
        int c = c0 + lane, dx = 0, dy = 0, dz = 0;
        if (r > 0 && c < faces) {  // the two faces across z
          dz = c < side * side ? -r : r;
          c = c < side * side ? c : c - side * side;
          dx = c % side - r;
          dy = c / side - r;
        } else if (r > 0 && c < cells) {  // the layers between them: four edges of 2 r cells
          c -= faces;
          dz = c / layer - (r - 1);
          const int edge = c % layer / (2 * r), o = c % (2 * r) - r;
          dx = edge == 0 ? o : (edge == 1 ? r : (edge == 2 ? -o : -r));
          dy = edge == 0 ? -r : (edge == 1 ? o : (edge == 2 ? r : -o));
        }
        const int qx = cx + dx, qy = cy + dy, qz = cz + dz;
        const float ex = fmaxf(fmaxf((float)qx - fx, fx - (float)(qx + 1)) - g.slack, 0.0f);
        const float ey = fmaxf(fmaxf((float)qy - fy, fy - (float)(qy + 1)) - g.slack, 0.0f);
        const float ez = fmaxf(fmaxf((float)qz - fz, fz - (float)(qz + 1)) - g.slack, 0.0f);
        uint32_t s = 0, len = 0;
        if (c0 + lane < cells && !((ex * ex + ey * ey + ez * ez) * g.s2_low > limit)) {
          const uint32_t b = bucket(g, qx, qy, qz);
          s = start[b];
          len = start[b + 1] - s;
        }
        const uint32_t tag = cell_tag(qx, qy, qz);
        for (unsigned m = __ballot_sync(0xffffffffu, len > 0u); m && scanned < kMaxScan; m &= m - 1u) {
          const int src = __ffs(m) - 1;
          const uint32_t first = __shfl_sync(0xffffffffu, s, src), want = __shfl_sync(0xffffffffu, tag, src);
          const uint32_t take = min(__shfl_sync(0xffffffffu, len, src), (uint32_t)(kMaxScan - scanned));
          scanned += (int)take;
          for (uint32_t t = lane; t < take; t += 32) {
            const float4 q = sorted[first + t];
            const float d2 = dist2(q.x - px, q.y - py, q.z - pz);
            if (d2 < best.d[K - 1] && __float_as_uint(q.w) == want && first + t != own) best.insert(d2);
          }
          __syncwarp();
        }
      }
      // the k-th smallest so far; the k smallest stay, one in each of the first k lanes
      float mine = INFINITY;
      for (int q = 0; q < k; ++q) {
        const uint32_t head = __float_as_uint(best.d[0]);
        const uint32_t least = __reduce_min_sync(0xffffffffu, head);
        const unsigned who = __ballot_sync(0xffffffffu, head == least);
        if (lane == __ffs(who) - 1) {
#pragma unroll
          for (int i = 0; i < K - 1; ++i) best.d[i] = best.d[i + 1];
          best.d[K - 1] = INFINITY;
        }
        kth = __uint_as_float(least);
        if (lane == q) mine = kth;
      }
      best.clear();
      best.d[0] = mine;
      limit = fminf(limit, kth * 1.00001f);
      const float reach = fmaxf((float)r - g.slack, 0.0f);
      if (kth <= reach * reach * g.s2_low || (float)r >= ball || scanned >= kMaxScan) break;
    }
    if (lane == 0) radius[at] = fminf(known, sqrtf(kth));
  }
}

struct Layout {
  size_t box, samples, bound, list_count, list, bkt, count, start, tiles, sorted, index, pending, total;
  int64_t m;            // buckets
  int64_t groups;       // groups of kSubGroup points in the samples' subset
  bool scan;            // the subset is not the whole cloud
};

size_t up(size_t v) { return (v + 255) / 256 * 256; }

Layout layout(int64_t n) {
  Layout L{};
  // in the median a search cell holds 4 (curves), 9 (surfaces) or 12 (volumes) points; a
  // bucket per two points keeps shared buckets rare (5M points of 50 surfaces 1.12 ms, 1.16
  // with one per four; 1M of 500 surfaces 0.68, 0.76)
  int64_t m = 256;
  while (m < n / 2) m <<= 1;
  L.m = m;
  const int64_t total = (n + kSubGroup - 1) / kSubGroup;
  L.groups = std::min(total, std::max((int64_t)kSubLeast / kSubGroup, total / 128));
  L.scan = L.groups < total;
  size_t o = 0;
  L.box = o;         o = up(o + 9 * 4);  // and Counts
  L.samples = o;     o = up(o + kSamples * 4);
  L.bound = o;       o = up(o + kSamples * 4);
  L.list_count = o;  o = up(o + kSamples * 4);
  L.list = o;        o = up(o + (L.scan ? (size_t)kSamples * kListCap * 4 : 0));
  L.bkt = o;         o = up(o + (size_t)n * 8);
  L.count = o;       o = up(o + (size_t)m * 4);
  L.start = o;       o = up(o + ((size_t)m + 1) * 4);
  L.tiles = o;       o = up(o + (size_t)((m + kScanTile - 1) / kScanTile) * 4);
  L.sorted = o;      o = up(o + (size_t)n * 16);
  L.index = o;       o = up(o + (size_t)n * 4);
  L.pending = o;     o = up(o + (size_t)n * 4);
  L.total = o;
  return L;
}

}  // namespace
}  // namespace knn
}  // namespace adop

using namespace adop::knn;

extern "C" {

size_t adop_point_radius_workspace_bytes(int64_t n) {
  if (n < 0 || n >= ((int64_t)1 << 31)) return 0;
  return layout(n < 1 ? 1 : n).total;
}

adop_status adop_point_radius(const float* xyz, int64_t n, int32_t k, float* radius, void* workspace,
                              size_t workspace_bytes, adop_stream stream) {
  auto fail = [](adop_status st, const char* msg) {
    adop::set_last_error(msg);
    return st;
  };
  if (n < 0 || n >= ((int64_t)1 << 31)) return fail(ADOP_ERR_INVALID_ARG, "point count outside [0, 2^31)");
  if (k < 1 || k > kMaxK) return fail(ADOP_ERR_INVALID_ARG, "k outside [1, 16]");
  if (n == 0) return ADOP_OK;
  if (!xyz || !radius) return fail(ADOP_ERR_INVALID_ARG, "xyz and radius must not be NULL");
  const Layout L = layout(n);
  if (workspace_bytes < L.total) return fail(ADOP_ERR_OUT_OF_MEMORY, "workspace too small for adop_point_radius");
  if (!workspace || ((uintptr_t)workspace & 255) != 0)
    return fail(ADOP_ERR_INVALID_ARG, "workspace must be a 256-byte aligned device pointer");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(workspace);
  uint32_t* box = reinterpret_cast<uint32_t*>(ws + L.box);
  float* samples = reinterpret_cast<float*>(ws + L.samples);
  float* bound = reinterpret_cast<float*>(ws + L.bound);
  uint32_t* list_count = reinterpret_cast<uint32_t*>(ws + L.list_count);
  float* list = reinterpret_cast<float*>(ws + L.list);
  uint2* bkt = reinterpret_cast<uint2*>(ws + L.bkt);
  uint32_t* count = reinterpret_cast<uint32_t*>(ws + L.count);
  uint32_t* start = reinterpret_cast<uint32_t*>(ws + L.start);
  uint32_t* tiles = reinterpret_cast<uint32_t*>(ws + L.tiles);
  float4* sorted = reinterpret_cast<float4*>(ws + L.sorted);
  uint32_t* index = reinterpret_cast<uint32_t*>(ws + L.index);
  uint32_t* pending = reinterpret_cast<uint32_t*>(ws + L.pending);
  const int blocks = adop::num_sms() * 8;
  cudaError_t e;
  if ((e = cudaMemsetAsync(box, 0xff, 3 * 4, s)) != cudaSuccess ||
      (e = cudaMemsetAsync(box + 3, 0, 6 * 4, s)) != cudaSuccess)
    return fail(ADOP_ERR_CUDA, cudaGetErrorString(e));
  k_bbox<<<blocks, 256, 0, s>>>(xyz, n, box);
  k_sample_bound<<<kSamples, kBoundThreads, 0, s>>>(xyz, n, k, L.groups, bound, list_count);
  if (L.scan)
    k_sample_scan<<<(unsigned)std::min((n + 1023) / 1024, (int64_t)blocks), 256, 0, s>>>(xyz, n, bound, list_count, list);
  k_sample_select<<<kSamples, 256, 0, s>>>(xyz, n, k, L.scan ? 1 : 0, bound, list_count, list, samples);
  uint32_t hbox[6];
  float hs[kSamples];
  if ((e = cudaMemcpyAsync(hbox, box, sizeof(hbox), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
      (e = cudaMemcpyAsync(hs, samples, sizeof(hs), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
      (e = cudaStreamSynchronize(s)) != cudaSuccess)
    return fail(ADOP_ERR_CUDA, cudaGetErrorString(e));
  auto unord = [](uint32_t o) {
    uint32_t b = (o & 0x80000000u) ? (o & 0x7fffffffu) : ~o;
    float f;
    memcpy(&f, &b, 4);
    return f;
  };
  float lo[3], hi[3];
  for (int d = 0; d < 3; ++d) {
    lo[d] = unord(hbox[d]);
    hi[d] = unord(hbox[3 + d]);
  }
  const float extent = std::max({hi[0] - lo[0], hi[1] - lo[1], hi[2] - lo[2], 0.0f});
  if (!std::isfinite(extent)) return fail(ADOP_ERR_INVALID_ARG, "non-finite point positions");
  std::vector<float> v;
  for (float x : hs)
    if (std::isfinite(x)) v.push_back(x);
  float h = 0.0f;
  if (!v.empty()) {
    std::nth_element(v.begin(), v.begin() + v.size() / 2, v.end());
    h = 1.5f * v[v.size() / 2];
  }
  // at least extent / 2^20 (bounded cell coordinates) and a tiny absolute floor
  h = std::max({h, extent / 1048576.0f, 1e-20f});
  if (v.empty()) h = std::max(extent, 1e-20f);  // fewer than k + 1 points
  const int max_ring = (int)std::ceil(extent / h) + 2;
  auto grid_of = [&](float cell) {  // the sorted cells' size
    // (the square stays finite: 0 x inf would compare as no bound at all)
    return Grid{lo[0], lo[1], lo[2], 1.0f / h, 1.0f / cell, std::min(cell * cell * 0.99998f, FLT_MAX),
                extent / cell * 5e-7f + 1e-6f, (uint32_t)(L.m - 1)};
  };
  const Grid g = grid_of(h * kSearch);
  if ((e = cudaMemsetAsync(count, 0, (size_t)L.m * 4, s)) != cudaSuccess) return fail(ADOP_ERR_CUDA, cudaGetErrorString(e));
  k_count<<<blocks, 256, 0, s>>>(xyz, n, g, bkt, count);
  const int64_t nt = (L.m + kScanTile - 1) / kScanTile;
  k_scan_tiles<<<(unsigned)nt, 1024, 0, s>>>(count, L.m, tiles);
  k_scan_sums<<<1, 1024, 0, s>>>(tiles, nt);
  k_scan_apply<<<(unsigned)nt, 1024, 0, s>>>(count, L.m, tiles, start, (uint32_t)n);
  k_scatter<<<blocks, 256, 0, s>>>(xyz, n, g, bkt, start, sorted, index);
  const unsigned qblocks = (unsigned)std::min((n + 255) / 256, (int64_t)blocks * 8);
  uint32_t* counts = box + 6;
  if (k == 4) {
    k_query<4><<<qblocks, 256, 0, s>>>(n, k, g, start, sorted, index, radius, pending, counts);
    k_query_far<4><<<blocks, 256, 0, s>>>(k, g, start, sorted, index, max_ring, radius, pending, counts);
  } else {
    k_query<kMaxK><<<qblocks, 256, 0, s>>>(n, k, g, start, sorted, index, radius, pending, counts);
    k_query_far<kMaxK><<<blocks, 256, 0, s>>>(k, g, start, sorted, index, max_ring, radius, pending, counts);
  }
  const float fine = std::max({h / kFine, extent / 1048576.0f, 1e-20f});
  Grid gf = grid_of(fine);
  float most = (float)(std::min(max_ring, kMaxRing) + 1) * (h / fine) + gf.slack;
  void* args[] = {(void*)&xyz, &n, &k, &gf, &most, &bkt, &count, (void*)&L.m, &tiles, &start, &sorted, &index, &radius,
                  &pending, &counts};
  const void* dense = k == 4 ? (const void*)k_query_dense<4> : (const void*)k_query_dense<kMaxK>;
  for (int grid = adop::num_sms() * kDenseBlocksPerSm;; grid /= 2) {  // (fewer where only a part of the SMs is ours)
    e = cudaLaunchCooperativeKernel(dense, dim3(grid), dim3(256), args, 0, s);
    if (e != cudaErrorCooperativeLaunchTooLarge || grid < 2) break;
    cudaGetLastError();
  }
  if (e != cudaSuccess) return fail(ADOP_ERR_CUDA, cudaGetErrorString(e));
  if ((e = cudaGetLastError()) != cudaSuccess) return fail(ADOP_ERR_CUDA, cudaGetErrorString(e));
  return ADOP_OK;
}

}  // extern "C"
