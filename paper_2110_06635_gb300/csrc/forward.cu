// Forward pass of the one-pixel point rasterizer (Sec. 3.1): a depth-only
// pass, an accumulate pass for the points that pass the fuzzy depth test and
// a per-pixel normalise pass (the three-pass structure of the paper's
// implementation details), preceded by a clear of the keys; between the first
// two a per-pixel pass seeds every sum with the pixel's nearest point.
//
// Work decomposition: blockIdx.y selects the camera; blocks stride over
// points (or pixels) with a grid of whole waves of the kernel's resident
// blocks over the GPU's SMs (stride_grid).
#include <cuda_runtime.h>

#include "launch.h"

namespace adop {

int num_sms() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 1;
  }
  return sms;
}

int point_blocks(int64_t n, int ncam) {
  const int64_t want = (n + kThreads - 1) / kThreads;
  const int64_t cap = ((int64_t)num_sms() * 8 + ncam - 1) / ncam;
  int64_t b = want < cap ? want : cap;
  return (int)(b < 1 ? 1 : b);
}

namespace {
// Resident blocks per SM of kernel k (occupancy calculator), cached per
// calling thread: a launch asks the runtime once per kernel and thread.
int resident_blocks(const void* k, size_t smem, int threads) {
  struct Entry {
    const void* k;
    size_t smem;
    int threads, n;
  };
  constexpr int kEntries = 256;
  static thread_local Entry cache[kEntries];
  static thread_local int used = 0;
  for (int i = 0; i < used; ++i)
    if (cache[i].k == k && cache[i].smem == smem && cache[i].threads == threads) return cache[i].n;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem) != cudaSuccess || n < 1) n = 1;
  if (used < kEntries) cache[used++] = Entry{k, smem, threads, n};
  return n;
}
}  // namespace

dim3 stride_grid(const void* k, int64_t work, int ncam, int waves, size_t smem, int threads) {
  const int64_t want = (work + threads - 1) / threads;
  const int64_t cap = ((int64_t)num_sms() * resident_blocks(k, smem, threads) * waves + ncam - 1) / ncam;
  const int64_t b = want < cap ? want : cap;
  return dim3((unsigned)(b < 1 ? 1 : b), (unsigned)ncam);
}

// ---------------------------------------------------------------------------
// clear: key = UINT64_MAX (empty) for every pixel and, unless the seed pass
// writes them (a.seeded), count = 0 and acc = 0
// ---------------------------------------------------------------------------
template <int C>
__global__ void __launch_bounds__(kThreads) k_clear(const __grid_constant__ LaunchCams cams,
                                                    const __grid_constant__ PointArgs a) {
  pdl_entry();
  const DevCam& cam = cams.c[blockIdx.y];
  const int64_t total = cam.off[a.levels];
  // a pixel's sums as 256-bit stores (one full sector each) where C % 8 == 0
  // and acc is 32-byte aligned -- the workspace's always is, a caller's frame
  // need only be 16-byte aligned (23.1 -> 22.2 us on the 1080p step)
  const bool v8 = (C % 8 == 0) && (((uintptr_t)cam.acc & 31u) == 0u);
  int lc = 0;  // the layer of g: g only grows, so its layer only advances
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total;
       g += (int64_t)gridDim.x * blockDim.x) {
    while (lc + 1 < a.levels && g >= cam.off[lc + 1]) ++lc;
    const int64_t p = g - cam.off[lc];
    cam.key[lc][p] = ~0ull;
    if (a.seeded) continue;
    cam.cnt[lc][p] = 0u;
    const float z[C] = {};
    if (v8) {
      store_row<C>(cam.acc + g * C, z);
    } else {
      store_vec<C>(cam.acc + g * C, z);
    }
  }
}

// ---------------------------------------------------------------------------
// K1 depth pass: key[l][p] = min over points of (bits(z) << 32 | i)
// One thread per point; the keys are read first and the 64-bit atomicMin is
// issued only where the point can still win (most points are occluded).
// Every layer's key is read before any atomic, so that the kL reads are in
// flight together rather than one round trip per layer (65.5 -> 60.2 us on
// the 1080p step).  (Measured on GB300: grouping lanes that share a pixel
// with __match_any_sync was 4x slower -- the per-group warp intrinsics
// serialise -- and interleaving two points per thread 25% slower.)
// The pass also records, per point, the layers where it may still pass the
// fuzzy test (cam.early, one byte): it cannot where its depth already exceeds
// f32(z_cur (1 + alpha)) for the key z_cur it read, since keys only decrease
// (z_cur >= the final z_min, and f32(. * (1 + alpha)) is monotone), so the
// accumulate pass's test would reject it there as well.  The accumulate
// pass skips those layers' key reads, and skips outright the points outside
// the view or behind at every layer (on the 120M-point frame, 70% of the
// points are outside the view: accumulate 770 -> 581 us, and 528 us once the
// position is read only for points with a layer left).
// ---------------------------------------------------------------------------
// One point at every layer.  kInside: the point is inside the image at every
// layer (in_every_layer), so no layer is tested.  kPlain: no discarding.
// Returns the layers where the point may still pass the fuzzy test.
template <int kL, bool kInside, bool kPlain>
__device__ __forceinline__ uint32_t depth_layers(const DevCam& cam, const PointArgs& a, float u0, float v0, float zd,
                                                 uint32_t i) {
  const bool discard = !kPlain && a.radius != nullptr;
  const float rw = discard ? __ldg(a.radius + i) : 0.0f, bt = discard ? __ldg(a.beta + i) : 0.0f;
  const int levels = kL < ADOP_MAX_LEVELS ? kL : a.levels;
  int32_t pix[kL];  // pixel within layer l (< 2^28), -1: none
#pragma unroll
  for (int l = 0; l < kL; ++l) {
    int32_t pu, pv;
    const bool in = pixel_in(u0, v0, l, cam.w, cam.h, pu, pv);
    pix[l] = pv * (cam.w >> l) + pu;
    if (!(kInside || in) || l >= levels || (discard && !discard_keep(cam, zd, rw, bt, a.g2, l))) pix[l] = -1;
  }
  // Only the upper half of a key, the depth, is read.  (An L1-cached read may
  // be stale, but keys only decrease: a stale value can cost an atomic that
  // loses, never skip one that wins, and it can only keep a layer in the mask
  // that a fresh value would have dropped.)
  uint32_t cur[kL];
#pragma unroll
  for (int l = 0; l < kL; ++l)
    cur[l] = pix[l] >= 0 ? __ldca(reinterpret_cast<const uint32_t*>(cam.key[l] + pix[l]) + 1) : 0u;
  uint32_t em = 0;
#pragma unroll
  for (int l = 0; l < kL; ++l) {
    // an empty pixel's depth reads as NaN, and nothing is behind it.  alpha >= 0:
    // what is behind the fuzzy threshold is behind the nearest point too
    if (pix[l] < 0 || zd > __fmul_rn(__uint_as_float(cur[l]), a.a1)) continue;
    em |= 1u << l;
    // (an equal depth may win by its index: the atomic decides)
    if (__float_as_uint(zd) <= cur[l]) atomicMin(cam.key[l] + pix[l], depth_key(zd, i));
  }
  return em;
}

template <int kL, bool kPlain>
__global__ void __launch_bounds__(kThreads) k_depth(const __grid_constant__ LaunchCams cams,
                                                    const __grid_constant__ PointArgs a) {
  pdl_entry();
  const DevCam& cam = cams.c[blockIdx.y];
  const float* __restrict__ xyz = cam.xyz;
  const uint32_t n = (uint32_t)cam.n, S = gridDim.x * blockDim.x;  // n < 2^31, S < 2^23: no wrap
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += S) {
    const float* q = xyz + 3 * (int64_t)i;
    float X0, X1, X2, u0, v0, zd;
    uint32_t em = 0;  // layers where the point may still pass the fuzzy test
    transform(cam, __ldg(q), __ldg(q + 1), __ldg(q + 2), X0, X1, X2);
    const bool ok = (kPlain ? camera_plain(cam, X0, X1, X2, u0, v0, zd) : camera(cam, X0, X1, X2, u0, v0, zd)) &&
                    zd > a.znear;
    if (ok && u0 >= -0.5f && u0 < cam.inside_u && v0 >= -0.5f && v0 < cam.inside_v) {
      if (kPlain || !(cam.normals && !normal_keep(cam, cam.normals, i, X0, X1, X2)))
        em = depth_layers<kL, true, kPlain>(cam, a, u0, v0, zd, i);
    } else if (ok && in_pyramid(u0, v0, cam.w, cam.h, a.levels)) {
      if (kPlain || !(cam.normals && !normal_keep(cam, cam.normals, i, X0, X1, X2)))
        em = depth_layers<kL, false, kPlain>(cam, a, u0, v0, zd, i);
    }
    if (cam.early) __stcs(cam.early + i, (uint8_t)em);
  }
}

// ---------------------------------------------------------------------------
// K1b seed: the nearest point of a pixel is in its Lambda whatever alpha is,
// and the key names it, so every pixel starts with that point's descriptor as
// its sum and a count of 1 -- plain, coalesced stores -- and the accumulate
// pass adds only the others.  They are few: 1.13 pairs in Lambda per non-empty
// pixel on the 5M-point 1080p view, 1.09 at 4K, 1.56 with 20M points at 1440 x
// 810.  Clearing the sums and adding every member with atomics cost the 4K
// view's accumulate pass 1.05 GB of DRAM reads, most of them of cleared sums.
// An empty pixel's sums are cleared where the caller keeps them
// (cam.keep_acc), and are otherwise never read.
// ---------------------------------------------------------------------------
template <int C, typename TF>
__global__ void __launch_bounds__(kThreads) k_seed(const __grid_constant__ LaunchCams cams,
                                                   const __grid_constant__ PointArgs a) {
  pdl_entry();
  const DevCam& cam = cams.c[blockIdx.y];
  const TF* feat = reinterpret_cast<const TF*>(cam.feat);
  const int64_t total = cam.off[a.levels];
  // a pixel's sums as 256-bit stores (one full sector each) where C % 8 == 0
  // and acc is 32-byte aligned -- the workspace's always is, a caller's frame
  // need only be 16-byte aligned
  const bool v8 = (C % 8 == 0) && (((uintptr_t)cam.acc & 31u) == 0u);
  const int64_t S = (int64_t)gridDim.x * blockDim.x;
  int lc = 0;  // the layer of g: g only grows, so its layer only advances
  // two pixels at a time: their key -> descriptor chains overlap
  for (int64_t g0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g0 < total; g0 += 2 * S) {
    int lu[2];
    unsigned long long key[2];
    float f[2][C];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t g = g0 + u * S;
      while (lc + 1 < a.levels && g >= cam.off[lc + 1]) ++lc;
      lu[u] = lc;
      key[u] = g < total ? cam.key[lc][g - cam.off[lc]] : ~0ull;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
#pragma unroll
      for (int k = 0; k < C; ++k) f[u][k] = 0.0f;
      if (key[u] != ~0ull) load_desc<C, TF>(feat, (int64_t)(uint32_t)key[u], a.log_desc, f[u]);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int64_t g = g0 + u * S;
      if (g >= total) break;
      const bool empty = key[u] == ~0ull;
      cam.cnt[lu[u]][g - cam.off[lu[u]]] = empty ? 0u : 1u;
      if (empty && !cam.keep_acc) continue;
      if (v8) {
        store_row<C>(cam.acc + g * C, f[u]);
      } else {
        store_vec<C>(cam.acc + g * C, f[u]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// K2 accumulate: the points with z <= f32(z_min * (1 + alpha)) that are not
// their pixel's nearest add their descriptor to the pixel's FP32 sum (float4
// vector atomics) and increment |Lambda|; every point's layer mask of passed
// tests is written for the backward pass, with the point's layer-0 screen
// tile in bits 8..31 (where the caller or a backward reads it: cam.vis).
//
// A warp takes 32, 64 or 128 consecutive points, reads the depth pass's layer
// bytes (cam.early) and lists the points with a layer left; those are then
// projected again and tested, one per lane, so that the points which the
// depth pass ruled out -- outside the view, or hidden when they were met --
// cost a byte and a mask entry and leave no lane idle (19 of 32 lanes were
// active per instruction with 20M points at 1440 x 810).  As in K1, every
// layer's key is read before the tests.
// ---------------------------------------------------------------------------
// Blocks of 128 threads: with 256 a block took 1024 points, and on 5M points the last
// of few waves ran on part of the SMs (66 us, 62 with 128; 64 need a spill or lose a
// fifth of the resident warps: 69).
constexpr int kPerLane = 4;
constexpr int kAccumThreads = 128;

// 12 resident blocks per SM (at most 40 registers) where that costs no spills,
// 10 with five layers, 8 with more; with 16 channels 8 (64 registers), 6 with
// more than five layers.  (Left to the compiler, 16 channels took 107 to 128
// registers, 4 blocks: frames of 1M points in random order at 640x480 took 88
// us, now 72; 8M at 1080p 330, 264.)
template <int C, int kL>
constexpr int accum_min_blocks() {
  return C > 8 ? (kL <= 5 ? 8 : 6) : (kL <= 4 ? 12 : (kL == 5 ? 10 : 8));
}

template <int C, typename TF, int kL>
__global__ void __launch_bounds__(kAccumThreads, accum_min_blocks<C, kL>())
    k_accum(const __grid_constant__ LaunchCams cams, const __grid_constant__ PointArgs a, const int per_lane) {
  pdl_entry();
  __shared__ uint16_t s_list[kAccumThreads / 32][32 * kPerLane];  // point within the chunk | layers << 8
  const DevCam& cam = cams.c[blockIdx.y];
  const TF* feat = reinterpret_cast<const TF*>(cam.feat);
  const float* __restrict__ xyz = cam.xyz;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint16_t* list = s_list[warp];
  const bool early = cam.early != nullptr;
  const bool vis16 = per_lane == kPerLane && ((uintptr_t)cam.vis & 15u) == 0u;
  const int64_t S = (int64_t)gridDim.x * (kAccumThreads / 32) * 32 * per_lane;
  // this lane's layer bytes of the chunk at `base` (0: nothing left, or no point)
  auto bytes_at = [&](int64_t base) -> uint32_t {
    const int64_t i = base + lane * per_lane;
    if (i >= cam.n) return 0u;
    if (!early) {
      const int64_t left = cam.n - i;
      return ~0u >> (8 * (4 - (int)(left < per_lane ? left : per_lane)));
    }
    if (per_lane == 1) return (uint32_t)__ldcs(cam.early + i);
    if (i + per_lane <= cam.n)
      return per_lane == 2 ? (uint32_t)__ldcs(reinterpret_cast<const uint16_t*>(cam.early + i))
                           : __ldcs(reinterpret_cast<const uint32_t*>(cam.early + i));
    uint32_t w = 0u;
    for (int u = 0; u < per_lane && i + u < cam.n; ++u) w |= (uint32_t)__ldcs(cam.early + i + u) << (8 * u);
    return w;
  };
  int64_t base = ((int64_t)blockIdx.x * (kAccumThreads / 32) + warp) * 32 * per_lane;
  uint32_t next = bytes_at(base);
  for (; base < cam.n; base += S) {
    const uint32_t em4 = next;
    next = bytes_at(base + S);  // one chunk ahead: its round trip overlaps this chunk's
    const int64_t i0 = base + lane * per_lane;
    if (cam.vis) {
      if (em4 == 0u && vis16 && i0 + kPerLane <= cam.n) {
        *reinterpret_cast<uint4*>(cam.vis + i0) = make_uint4(0u, 0u, 0u, 0u);
      } else {
        for (int u = 0; u < per_lane; ++u)
          if (((em4 >> (8 * u)) & 0xFFu) == 0u && i0 + u < cam.n) cam.vis[i0 + u] = 0u;
      }
    }
    int total = 32;
    if (per_lane > 1) {  // list the points with a layer left, in order
      int slot = 0;
      total = 0;
#pragma unroll
      for (int u = 0; u < kPerLane; ++u) {
        const unsigned b = __ballot_sync(0xffffffffu, ((em4 >> (8 * u)) & 0xFFu) != 0u);
        slot += __popc(b & ((1u << lane) - 1u));
        total += __popc(b);
      }
      if (total == 0) continue;
#pragma unroll
      for (int u = 0; u < kPerLane; ++u) {
        const uint32_t em = (em4 >> (8 * u)) & 0xFFu;
        if (em) list[slot++] = (uint16_t)((uint32_t)(lane * per_lane + u) | (em << 8));
      }
      __syncwarp();
    }
    for (int r = lane; r < total; r += 32) {
      const uint32_t item = per_lane > 1 ? list[r] : ((uint32_t)lane | (em4 << 8));
      const uint32_t em = item >> 8;
      if (em == 0u) continue;  // (one point a lane)
      const int64_t i = base + (item & 0xFFu);
      uint32_t mask = 0;  // bit l: the point is in Lambda of its layer-l pixel
      // the forward's last read of the position is streamed (evict-first), so
      // that the pixel state keeps its place in L2
      const float x0 = __ldcs(xyz + 3 * i), x1 = __ldcs(xyz + 3 * i + 1), x2 = __ldcs(xyz + 3 * i + 2);
      float X0, X1, X2, u0 = 0.0f, v0 = 0.0f, zd;
      transform(cam, x0, x1, x2, X0, X1, X2);
      bool ok = camera(cam, X0, X1, X2, u0, v0, zd);
      // a layer bit of the depth pass stands for all of these tests
      if (!early)
        ok = ok && (zd > a.znear) && in_pyramid(u0, v0, cam.w, cam.h, a.levels) &&
             !(cam.normals && !normal_keep(cam, cam.normals, i, X0, X1, X2));
      if (ok) {
        const bool discard = !early && a.radius != nullptr;
        const float rw = discard ? __ldg(a.radius + i) : 0.0f, bt = discard ? __ldg(a.beta + i) : 0.0f;
        int32_t pix[kL];  // pixel within layer l (< 2^28), -1: none
        uint32_t zb[kL];
        uint32_t seeded = 0;  // the layers where the point is the pixel's nearest
#pragma unroll
        for (int l = 0; l < kL; ++l) {
          int32_t pu, pv;
          const bool keep = ((em >> l) & 1u) && l < a.levels && (!discard || discard_keep(cam, zd, rw, bt, a.g2, l));
          pix[l] = (keep && pixel_in(u0, v0, l, cam.w, cam.h, pu, pv)) ? pv * (cam.w >> l) + pu : -1;
        }
#pragma unroll
        for (int l = 0; l < kL; ++l) {
          const unsigned long long key = pix[l] >= 0 ? __ldg(cam.key[l] + pix[l]) : 0ull;
          zb[l] = (uint32_t)(key >> 32);
          if (a.seeded && (uint32_t)key == (uint32_t)i) seeded |= 1u << l;
        }
        float f[C];
        bool loaded = false;
#pragma unroll
        for (int l = 0; l < kL; ++l) {
          if (pix[l] < 0 || !(zd <= __fmul_rn(__uint_as_float(zb[l]), a.a1))) continue;
          mask |= 1u << l;
          if ((seeded >> l) & 1u) continue;
          if (!loaded) {
            load_feat_last<C, TF>(feat, i, f);
            if (a.log_desc) {
#pragma unroll
              for (int k = 0; k < C; ++k) f[k] = expf(f[k]);
            }
            loaded = true;
          }
          atomic_add_vec<C>(cam.acc + (cam.off[l] + pix[l]) * C, f);
          atomicAdd(cam.cnt[l] + pix[l], 1u);
        }
      }
      if (cam.vis) {
        uint32_t tile = 0;
        if (mask) {  // layer-0 screen tile of the point (position clamped to the image)
          const int32_t tu = min(max(__float2int_rn(u0), 0), cam.w - 1) >> kTileShift;
          const int32_t tv = min(max(__float2int_rn(v0), 0), cam.h - 1) >> kTileShift;
          tile = (uint32_t)(tv * cam.tiles_x + tu);
        }
        cam.vis[i] = (tile << 8) | mask;
      }
    }
    if (per_lane > 1) __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// K3 normalise: I = sum / |Lambda| (Eq. blend), background where empty (k_env_fill
// writes the environment map's pixels),
// photometric epilogue on layer 0, cast to the output type, planar layout
// ---------------------------------------------------------------------------
template <int C, typename TO>
__global__ void __launch_bounds__(kThreads) k_normalize(const __grid_constant__ LaunchCams cams,
                                                        const __grid_constant__ PointArgs a) {
  pdl_entry();
  const DevCam& cam = cams.c[blockIdx.y];
  const int64_t total = cam.off[a.levels];
  int lc = 0;  // the layer of g: g only grows, so its layer only advances
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total;
       g += (int64_t)gridDim.x * blockDim.x) {
    while (lc + 1 < a.levels && g >= cam.off[lc + 1]) ++lc;
    const int l = lc;
    TO* img = reinterpret_cast<TO*>(cam.image[l]);
    if (img == nullptr) continue;
    const int64_t p = g - cam.off[l];
    const int64_t np = cam.off[l + 1] - cam.off[l];
    // the count and the sums are loaded together: one round trip per pixel
    const uint32_t n = cam.cnt[l][p];
    float v[C];
    load_vec<C>(cam.acc + g * C, v);
    if (n == 0) {
      if (a.env) continue;  // the environment map's pixels: k_env_fill
#pragma unroll
      for (int k = 0; k < C; ++k) v[k] = a.background ? __ldg(a.background + k) : 0.0f;
    } else {  // one reciprocal per pixel (within 2 ulp of the quotient)
      const float rn = __frcp_rn((float)n);
#pragma unroll
      for (int k = 0; k < C; ++k) v[k] *= rn;
    }
    if (l == 0 && cam.epi) {
      const int32_t pu = (int32_t)(p % cam.w), pv = (int32_t)(p / cam.w);
#pragma unroll
      for (int k = 0; k < (C < 3 ? C : 3); ++k) v[k] = epilogue(cam, k, pu, pv, v[k], nullptr);
    }
#pragma unroll
    for (int k = 0; k < C; ++k) img[k * np + p] = from_f32<TO>(v[k]);
  }
}

int64_t most_pixels(const LaunchCams& cams, const PointArgs& a) {
  int64_t most = 0;
  for (int k = 0; k < a.ncam; ++k) most = cams.c[k].off[a.levels] > most ? cams.c[k].off[a.levels] : most;
  return most;
}

cudaError_t launch_clear(const LaunchCams& cams, const PointArgs& a, int c, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  const int64_t px = most_pixels(cams, a);
  ADOP_DISPATCH_C(c, e = launch_strided(k_clear<kC>, px, a.ncam, kPixelWaves, 0, s, cams, a));
  return e;
}

cudaError_t launch_seed(const LaunchCams& cams, const PointArgs& a, int c, adop_dtype fd, cudaStream_t s) {
  if (!a.seeded) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  const int64_t px = most_pixels(cams, a);
  ADOP_DISPATCH_C(c, ADOP_DISPATCH_T(fd, TF, e = launch_strided(k_seed<kC, TF>, px, a.ncam, kPixelWaves, 0, s, cams,
                                                                a)));
  return e;
}

// The seed pass pays once the cleared sums would not stay in the L2 (129 MB)
// until the atomics reach them: from 96 MB of pixel state over the launch's
// cameras (clear + seed + accumulate, us; 2.75M pixels of 1080p, 11M at 4K).
//   C = 4,  77 MB, 2.6M points:   70 without,   80 with
//   C = 8, 121 MB, 2.6M points:  106 without,  101 with
//   C = 8, 121 MB, 5M points:    116 without,  111 with
//   C = 4, 308 MB, 120M points:  808 without,  573 with
// (Requiring a point per two pixels as well made the 1080p step of 1.2M points
// slower, 270 -> 277 us.)
// A kept state is written whole either way, the sums of empty pixels too; there
// the pass pays only with a point per 32 pixels (C = 8, step, with / without: 50
// thousand points at 1080p 161 / 154, 500 thousand 210 / 214; at 3000x2250 50
// thousand 384 / 371, 500 thousand 473 / 497).
int seed_rule(const LaunchCams& cams, const PointArgs& a, int c) {
  int64_t px = 0, kept = 0, points = 0;
  for (int k = 0; k < a.ncam; ++k) {
    const DevCam& cam = cams.c[k];
    px += cam.off[a.levels];
    kept += cam.keep_acc ? cam.off[a.levels] : 0;
    points += cam.n;
  }
  return px * (12 + 4 * (int64_t)c) >= ((int64_t)96 << 20) && 32 * points >= kept ? 1 : 0;
}

int64_t most_points(const LaunchCams& cams, const PointArgs& a) {
  int64_t most = 0;
  for (int k = 0; k < a.ncam; ++k) most = cams.c[k].n > most ? cams.c[k].n : most;
  return most;
}

cudaError_t launch_depth(const LaunchCams& cams, const PointArgs& a, cudaStream_t s) {
  const int64_t n = most_points(cams, a);
  if (n == 0) return cudaSuccess;
  bool plain = a.radius == nullptr;
  for (int k = 0; k < a.ncam; ++k) plain = plain && !cams.c[k].normals && camera_is_plain(cams.c[k]);
#define ADOP_DEPTH(L)                                                                       \
  return plain ? launch_strided(k_depth<L, true>, n, a.ncam, kPointWaves, 0, s, cams, a)    \
               : launch_strided(k_depth<L, false>, n, a.ncam, kPointWaves, 0, s, cams, a)
  switch (a.levels) {
    case 1: ADOP_DEPTH(1);
    case 2: ADOP_DEPTH(2);
    case 3: ADOP_DEPTH(3);
    case 4: ADOP_DEPTH(4);
    case 5: ADOP_DEPTH(5);
    default: ADOP_DEPTH(ADOP_MAX_LEVELS);
  }
#undef ADOP_DEPTH
}

cudaError_t launch_accum(const LaunchCams& cams, const PointArgs& a, int c, adop_dtype fd, cudaStream_t s) {
  const int64_t n = most_points(cams, a);
  if (n == 0) return cudaSuccess;
  // four points a lane where that leaves 2.5 waves of resident warps, else two
  // or one, which skip less but fill the last wave (C = 4 at 1080p, us with
  // 1 / 2 / 4 a lane: 400 thousand points 19.0 / 20.7 / 21.6, 1.2M 28.9 / 29.5 /
  // 32.9, 3.5M 52.5 / 50.0 / 49.9, 8M 92.8 / 82.0 / 77.9, in random order 127 / 96 / 87)
  int per_lane = kPerLane;
  while (per_lane > 1 && 2 * n * a.ncam < 5 * (int64_t)num_sms() * 48 * 32 * per_lane) per_lane /= 2;
  const int64_t work = (n + per_lane - 1) / per_lane;
  cudaError_t e = cudaSuccess;
#define ADOP_ACCUM(L)                                                                                       \
  ADOP_DISPATCH_C(c, ADOP_DISPATCH_T(fd, TF, e = launch_pdl(k_accum<kC, TF, L>,                             \
      stride_grid((const void*)k_accum<kC, TF, L>, work, a.ncam, kPointWaves, 0, kAccumThreads),            \
      dim3(kAccumThreads), 0, s, cams, a, per_lane)))
  if (a.levels <= 4) {
    ADOP_ACCUM(4);
  } else if (a.levels == 5) {
    ADOP_ACCUM(5);
  } else {
    ADOP_ACCUM(ADOP_MAX_LEVELS);
  }
#undef ADOP_ACCUM
  return e;
}

cudaError_t launch_normalize(const LaunchCams& cams, const PointArgs& a, int c, adop_dtype od, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  const int64_t px = most_pixels(cams, a);
  ADOP_DISPATCH_C(c, ADOP_DISPATCH_T(od, TO, e = launch_strided(k_normalize<kC, TO>, px, a.ncam, kPixelWaves, 0, s,
                                                                cams, a)));
  return e;
}

}  // namespace adop
