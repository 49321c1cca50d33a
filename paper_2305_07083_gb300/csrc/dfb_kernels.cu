// CUDA kernels of the DFB path for sm_103a, apart from the composite kernel
// (dfb_composite.cu):
//
//   K1  bucket:     per-tile lists (grouped by the host) sorted by (order key,
//                   submit index): the rank order of the list tree (Sec. 4.2)
//                   and the tile blocks the composite reads.
//   K6  convert:    producer-side FP16 / BF16 / FP8-e4m3 storage of tiles.
//   read-back:      normalised accumulation and per-pixel variance.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "dfb_device.cuh"
#include "dfb_internal.h"

namespace dfb {

// ----------------------------------------------------------------------------
// K1: bucketing
// ----------------------------------------------------------------------------
// Lists longer than this are sorted with a bitonic network in shared memory
// (one warp per tile); longer ones than kSortSmem by rank counting.
constexpr int kOrderWarps = 8;
constexpr int kSortSmem = 256;

// One warp per tile.  The tile's records arrive grouped, in submission order;
// the element at position i gets the key (order-key bits << 32 | i), and its
// final place is its rank under that key: the (key, submit index) order.
// Lists of up to 32 are ranked in registers, longer ones sorted in shared
// memory.
__device__ __forceinline__ void order_tile(const FragRec* grouped, const int* tileOff, int t,
                                           FragRec* __restrict__ srecs,
                                           TileBlock* __restrict__ blocks, uint64_t* a, int lane) {
  const int off = tileOff[t];
  const int n = tileOff[t + 1] - off;
  if (lane == 0) {
    blocks[t].n = n;
    blocks[t].off = off;
  }
  const FragRec* in = grouped + off;
  if (n <= 32) {
    FragRec r{};
    uint64_t k = ~0ull;
    if (lane < n) {
      r = in[lane];
      k = ((uint64_t)r.key << 32) | (uint32_t)lane;
    }
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += (__shfl_sync(0xffffffffu, k, j) < k) ? 1 : 0;
    if (lane < n) {
      srecs[off + rank] = r;
      if (rank < kStageFragments) blocks[t].recs[rank] = r;
    }
    return;
  }
  if (n <= kSortSmem) {
    int m = 64;
    while (m < n) m <<= 1;
    for (int i = lane; i < m; i += 32)
      a[i] = i < n ? (((uint64_t)in[i].key << 32) | (uint32_t)i) : ~0ull;
    __syncwarp();
    for (int k = 2; k <= m; k <<= 1) {
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int i = lane; i < m; i += 32) {
          const int p = i ^ j;
          if (p > i) {
            const uint64_t x = a[i], y = a[p];
            const bool up = (i & k) == 0;
            if ((x > y) == up) {
              a[i] = y;
              a[p] = x;
            }
          }
        }
        __syncwarp();
      }
    }
    for (int i = lane; i < n; i += 32) {
      const FragRec r = in[(uint32_t)a[i]];
      srecs[off + i] = r;
      if (i < kStageFragments) blocks[t].recs[i] = r;
    }
    return;
  }
  // very long lists: rank of each element by counting the smaller keys
  for (int jb = 0; jb < n; jb += 32) {
    const int j = jb + lane;
    const uint64_t kj = j < n ? (((uint64_t)in[j].key << 32) | (uint32_t)j) : ~0ull;
    int rank = 0;
    for (int mb = 0; mb < n; mb += 32) {
      const int m = mb + lane;
      const uint64_t km = m < n ? (((uint64_t)in[m].key << 32) | (uint32_t)m) : ~0ull;
      const int cnt = min(32, n - mb);
      for (int q = 0; q < cnt; ++q) rank += (__shfl_sync(0xffffffffu, km, q) < kj) ? 1 : 0;
    }
    if (j < n) {
      const FragRec r = in[j];
      srecs[off + rank] = r;
      if (rank < kStageFragments) blocks[t].recs[rank] = r;
    }
  }
}

__global__ void __launch_bounds__(kOrderWarps * 32) k1_order(const FragRec* __restrict__ grouped,
                                                            const int* __restrict__ tileOff,
                                                            int nTiles, FragRec* __restrict__ srecs,
                                                            TileBlock* __restrict__ blocks,
                                                            int* __restrict__ redo) {
  __shared__ uint64_t keys[kOrderWarps][kSortSmem];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * kOrderWarps + warp;
  if (redo && blockIdx.x == 0 && threadIdx.x == 0) redo[0] = 0;
  if (t < nTiles) order_tile(grouped, tileOff, t, srecs, blocks, keys[warp], lane);
}

// A small frame's records come with the launch itself.  An upload, a launch
// on a side stream and the events between the streams cost the host more
// than such a frame takes on the GPU; here the bucketing is one more launch
// on the frame's own stream.
__global__ void __launch_bounds__(kOrderWarps * 32)
    k1_order_inline(const __grid_constant__ InlineFrame frame, FrameHeader* __restrict__ hdr,
                    FragRec* __restrict__ srecs, TileBlock* __restrict__ blocks,
                    int* __restrict__ redo) {
  __shared__ uint64_t keys[kOrderWarps][kSortSmem];
  grid_dependency_wait();  // an earlier frame may still read the buffers
  allow_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * kOrderWarps + warp;
  if (blockIdx.x == 0) {
    if (redo && threadIdx.x == 0) redo[0] = 0;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(&frame.hdr);
    for (int i = threadIdx.x; i < (int)(sizeof(FrameHeader) / 4); i += kOrderWarps * 32)
      reinterpret_cast<uint32_t*>(hdr)[i] = src[i];
  }
  if (t < frame.nTiles)
    order_tile(frame.recs, frame.tileOff, t, srecs, blocks, keys[warp], lane);
}

cudaError_t launch_bucket(const FragRec* grouped, const int* tileOff, int nTiles, FragRec* srecs,
                          TileBlock* blocks, int* redo, cudaStream_t s) {
  const int grid = nTiles > 0 ? (nTiles + kOrderWarps - 1) / kOrderWarps : 1;
  k1_order<<<grid, kOrderWarps * 32, 0, s>>>(grouped, tileOff, nTiles, srecs, blocks, redo);
  return cudaGetLastError();
}

cudaError_t launch_bucket_inline(const InlineFrame& frame, FrameHeader* hdr, FragRec* srecs,
                                 TileBlock* blocks, int* redo, cudaStream_t s) {
  static_assert(sizeof(FrameHeader) % 4 == 0, "copied by words");
  const int grid = frame.nTiles > 0 ? (frame.nTiles + kOrderWarps - 1) / kOrderWarps : 1;
  return launch_programmatic(k1_order_inline, grid, kOrderWarps * 32, 0, s, frame, hdr, srecs,
                             blocks, redo);
}

// ----------------------------------------------------------------------------
// read-back helpers
// ----------------------------------------------------------------------------
// Device read-backs follow a frame's kernels and one another on its stream.
// They are launched programmatically, so that each starts while the one
// before it drains (a copy would wait for the drain and start anew): four
// 1920x1080 passes that read their mean and variance images 371 -> 337 us, 16
// mixed frames with their colour and RGBA8 images 988 -> 915 us.  The kernels
// themselves are at HBM speed.  Frames hold at most 2^31 pixels.
__global__ void k_tiles_to_image(const float4* __restrict__ a, const float4* __restrict__ b,
                                 float scale, float4* __restrict__ out, int W, int H, int T,
                                 int logT, int tilesX) {
  grid_dependency_wait();
  allow_dependents();
  const uint32_t n = (uint32_t)W * (uint32_t)H;
  for (uint64_t i64 = blockIdx.x * blockDim.x + threadIdx.x; i64 < n;
       i64 += gridDim.x * blockDim.x) {
    const uint32_t i = (uint32_t)i64;
    const uint32_t y = i / (uint32_t)W, x = i - y * (uint32_t)W;
    const int64_t src = ((int64_t)(y >> logT) * tilesX + (x >> logT)) * ((int64_t)T * T) +
                        ((y & (T - 1)) << logT) + (x & (T - 1));
    float4 v = a[src];
    if (b) {
      const float4 c = b[src];
      v = make_float4(v.x - c.x, v.y - c.y, v.z - c.z, v.w - c.w);
    }
    // evict-first in L2: an accumulation that is read after every pass keeps
    // more of its state there (four 1920x1080 passes 337 -> 324 us)
    __stcs(out + i, make_float4(v.x * scale, v.y * scale, v.z * scale, v.w * scale));
  }
}

// n 32-bit words, src and dst 16-byte aligned; 64 bytes per thread in flight.
constexpr int kCopySpan = 4;
__global__ void __launch_bounds__(256) k_copy(const uint32_t* __restrict__ src,
                                              uint32_t* __restrict__ dst, size_t n) {
  grid_dependency_wait();
  allow_dependents();
  const size_t n4 = n >> 2;
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
  uint4* d4 = reinterpret_cast<uint4*>(dst);
  const size_t i0 = (size_t)blockIdx.x * (256 * kCopySpan) + threadIdx.x;
  uint4 v[kCopySpan];
#pragma unroll
  for (int u = 0; u < kCopySpan; ++u)
    if (i0 + 256 * u < n4) v[u] = s4[i0 + 256 * u];
#pragma unroll
  for (int u = 0; u < kCopySpan; ++u)
    if (i0 + 256 * u < n4) d4[i0 + 256 * u] = v[u];
  if (blockIdx.x == 0 && threadIdx.x < (n & 3)) dst[4 * n4 + threadIdx.x] = src[4 * n4 + threadIdx.x];
}

__global__ void k_image_to_tiles(const float4* __restrict__ in, float4* __restrict__ out, int W,
                                 int H, int T, int logT, int tilesX) {
  const int64_t n = (int64_t)W * H;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int y = (int)(i / W), x = (int)(i - (int64_t)y * W);
    const int64_t dst = ((int64_t)(y >> logT) * tilesX + (x >> logT)) * ((int64_t)T * T) +
                        ((y & (T - 1)) << logT) + (x & (T - 1));
    out[dst] = in[i];
  }
}

static int grid_for(int64_t n) {
  int64_t g = (n + 255) / 256;
  return (int)(g > 4096 ? 4096 : (g < 1 ? 1 : g));
}

static int log2_of(int T) {
  int l = 0;
  while ((1 << l) < T) ++l;
  return l;
}

cudaError_t launch_tiles_to_image(const float4* a, const float4* b, float scale, float4* out,
                                  int W, int H, int T, cudaStream_t s) {
  return launch_programmatic(k_tiles_to_image, grid_for((int64_t)W * H), 256, 0, s, a, b, scale,
                             out, W, H, T, log2_of(T), (W + T - 1) / T);
}

cudaError_t launch_copy(const uint32_t* src, uint32_t* dst, size_t words, cudaStream_t s) {
  const size_t blocks = (words / 4 + 256 * kCopySpan - 1) / (256 * kCopySpan);
  return launch_programmatic(k_copy, (int)(blocks ? blocks : 1), 256, 0, s, src, dst, words);
}

cudaError_t launch_image_to_tiles(const float4* in, float4* out, int W, int H, int T,
                                  cudaStream_t s) {
  k_image_to_tiles<<<grid_for((int64_t)W * H), 256, 0, s>>>(in, out, W, H, T, log2_of(T),
                                                            (W + T - 1) / T);
  return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// K6: producer-side storage conversion
// ----------------------------------------------------------------------------
// FP16 / BF16.  Bound by HBM: 6 bytes per value.  Every thread converts
// kHalfSpan groups of 8 values: two 16-byte loads and one 16-byte store per
// group, all loads issued before the first store, so that 64 KB per SM and
// more are in flight.  2,313 tiles of 64x64: 36.4 us, 6.25 TB/s (one value per
// load and 2-byte stores took 41.8 us).
constexpr int kHalfSpan = 2;

__device__ __forceinline__ uint32_t two_halves(float lo, float hi, __half) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t two_halves(float lo, float hi, __nv_bfloat16) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ __half to_half(float x, __half) { return __float2half_rn(x); }
__device__ __forceinline__ __nv_bfloat16 to_half(float x, __nv_bfloat16) {
  return __float2bfloat16_rn(x);
}

// src and dst 16-byte aligned; the last n % 8 values are converted singly.
template <class H>
__global__ void __launch_bounds__(256) k_to_half(const float* __restrict__ src, H* __restrict__ dst,
                                                 int64_t n) {
  const int64_t groups = n >> 3;
  const float4* s4 = reinterpret_cast<const float4*>(src);
  uint4* d4 = reinterpret_cast<uint4*>(dst);
  const int64_t g0 = (int64_t)blockIdx.x * (256 * kHalfSpan) + threadIdx.x;
  float4 lo[kHalfSpan], hi[kHalfSpan];
#pragma unroll
  for (int u = 0; u < kHalfSpan; ++u)
    if (g0 + 256 * u < groups) {
      lo[u] = __ldcs(s4 + 2 * (g0 + 256 * u));
      hi[u] = __ldcs(s4 + 2 * (g0 + 256 * u) + 1);
    }
#pragma unroll
  for (int u = 0; u < kHalfSpan; ++u)
    if (g0 + 256 * u < groups)
      d4[g0 + 256 * u] =
          make_uint4(two_halves(lo[u].x, lo[u].y, H()), two_halves(lo[u].z, lo[u].w, H()),
                     two_halves(hi[u].x, hi[u].y, H()), two_halves(hi[u].z, hi[u].w, H()));
  if (blockIdx.x == 0 && threadIdx.x < (n & 7)) {
    const int64_t i = (groups << 3) + threadIdx.x;
    dst[i] = to_half(src[i], H());
  }
}

// Any alignment, one value at a time.
template <class H>
__global__ void k_to_half_any(const float* __restrict__ src, H* __restrict__ dst, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = to_half(src[i], H());
}

template <class H>
void launch_half(const float* src, H* dst, int64_t n, cudaStream_t s) {
  const int64_t blocks = (n / 8 + 256 * kHalfSpan - 1) / (256 * kHalfSpan);
  if (((uintptr_t)src | (uintptr_t)dst) % 16 || blocks > 0x7fffffff)
    k_to_half_any<H><<<grid_for(n), 256, 0, s>>>(src, dst, n);
  else
    k_to_half<H><<<(int)(blocks ? blocks : 1), 256, 0, s>>>(src, dst, n);
}

// FP8: amax of the tile, scale = amax / 448 (1 for an all-zero tile), then
// code = e4m3(x / scale) with round-to-nearest-even and saturation.
__device__ __forceinline__ float fp8_scale(float amax) {
  return amax > 0.0f ? __fdiv_rn(amax, 448.0f) : 1.0f;
}
// x / s rounded to nearest, for r = 1 / s rounded to nearest and s in
// [2^-60, 2^60]: the quotient estimate x * r is corrected twice by its exact
// residual (P. Markstein, "Computation of elementary functions on the IBM RISC
// System/6000 processor", IBM J. Res. Dev. 34(1), 1990: the first correction
// makes it faithful, the second correctly rounded).  The residual is exact
// for |x| >= 2^-100; a smaller x gives a quotient below 2^-40, whose e4m3
// code is a signed zero whatever its last bits are.  The division proper
// takes a slow path for a zero dividend, and the pixels a fragment leaves
// empty are zeros.
__device__ __forceinline__ float fp8_quotient(float x, float s, float r) {
  float q = x * r;
  q = fmaf(fmaf(-q, s, x), r, q);
  q = fmaf(fmaf(-q, s, x), r, q);
  return copysignf(q, x);  // keeps the sign of a zero
}
__device__ __forceinline__ uint32_t fp8_two(float lo, float hi) {
  unsigned short two;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(two) : "f"(hi), "f"(lo));
  return two;
}
__device__ __forceinline__ float abs_max(float m, float4 v) {
  return fmaxf(fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
}

// The scale is known only once the whole tile has been read, so the tile
// stays in registers in between: TPT threads hold a tile of 32 * TPT values,
// 8 float4 each, loaded before the first is looked at, and every value is
// read from memory once.  A CTA of 512 threads holds 512 / TPT tiles (T = 4
// to 64: 2 to 512 threads per tile); a tile of 128x128 is shared by a cluster
// of CL = 4 CTAs, which exchange their maxima through distributed shared
// memory.  src and dst 16-byte aligned.  5,585 tiles of 64x64: 70.7 us, 6.47 TB/s,
// bound by HBM (164.7 us with one CTA reading its tile twice, and as much with
// a division proper per value).  256x256 tiles, other sizes and unaligned
// pools take the general kernel below.
constexpr int kFp8Threads = 512;
constexpr int kFp8Per = 32;  // values per thread

template <int TPT, int CL>
__global__ void __launch_bounds__(kFp8Threads) k_to_fp8_tiles(const float* __restrict__ src,
                                                              uint8_t* __restrict__ dst,
                                                              float* __restrict__ scales,
                                                              int nTiles) {
  static_assert(CL == 1 || TPT == kFp8Threads * CL, "a cluster holds one tile");
  __shared__ float red[kFp8Threads / 32];
  __shared__ float clusterRed;
  constexpr int IN = TPT < kFp8Threads ? TPT : kFp8Threads;  // threads of a tile in this CTA
  constexpr int tiles = kFp8Threads / IN;                    // tiles (or part of one) per CTA
  const int part = CL == 1 ? 0 : (int)(blockIdx.x % CL);
  const int sub = threadIdx.x / IN, t = threadIdx.x % IN;
  const int64_t tile = CL == 1 ? (int64_t)blockIdx.x * tiles + sub : blockIdx.x / CL;
  const bool live = tile < nTiles;
  constexpr int V = kFp8Per / 4;
  const size_t base = (size_t)(live ? tile : 0) * (TPT * V) + (size_t)part * (IN * V) + t;
  const float4* s4 = reinterpret_cast<const float4*>(src) + base;
  float4 v[V];
#pragma unroll
  for (int u = 0; u < V; ++u) v[u] = live ? __ldcs(s4 + u * IN) : make_float4(0.f, 0.f, 0.f, 0.f);
  float m = 0.0f;
#pragma unroll
  for (int u = 0; u < V; ++u) m = abs_max(m, v[u]);
#pragma unroll
  for (int o = (IN < 32 ? IN : 32) / 2; o > 0; o >>= 1)
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (IN > 32) {
    constexpr int W = IN / 32;  // warps of a tile in this CTA
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    m = red[sub * W];
#pragma unroll
    for (int w = 1; w < W; ++w) m = fmaxf(m, red[sub * W + w]);
  }
  if (CL > 1) {
    if (threadIdx.x == 0) clusterRed = m;
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
    const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&clusterRed);
#pragma unroll
    for (int r = 0; r < CL; ++r) {
      uint32_t at;
      float other;
      asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(mine), "r"(r));
      asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(other) : "r"(at) : "memory");
      m = fmaxf(m, other);
    }
    // a CTA's shared memory stays until every CTA of the cluster has read it
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
  }
  if (!live) return;
  const float scale = fp8_scale(m);
  if (t == 0 && part == 0) scales[tile] = scale;
  uint32_t* d = reinterpret_cast<uint32_t*>(dst) + base;
  if (scale >= 0x1p-60f && scale <= 0x1p60f) {
    const float r = __frcp_rn(scale);
#pragma unroll
    for (int u = 0; u < V; ++u)
      d[u * IN] = fp8_two(fp8_quotient(v[u].x, scale, r), fp8_quotient(v[u].y, scale, r)) |
                  (fp8_two(fp8_quotient(v[u].z, scale, r), fp8_quotient(v[u].w, scale, r)) << 16);
  } else {
#pragma unroll 1
    for (int u = 0; u < V; ++u) {
      const float4 x = s4[u * IN];
      d[u * IN] = fp8_two(__fdiv_rn(x.x, scale), __fdiv_rn(x.y, scale)) |
                  (fp8_two(__fdiv_rn(x.z, scale), __fdiv_rn(x.w, scale)) << 16);
    }
  }
}

// Any tile size and alignment: one CTA per tile, the tile read twice.
__global__ void __launch_bounds__(256) k_to_fp8(const float* __restrict__ src,
                                                uint8_t* __restrict__ dst,
                                                float* __restrict__ scales, int tileVals) {
  __shared__ float red[8];
  const float* s = src + (size_t)blockIdx.x * tileVals;
  uint8_t* d = dst + (size_t)blockIdx.x * tileVals;
  float m = 0.0f;
  for (int i = threadIdx.x; i < tileVals; i += 256) m = fmaxf(m, fabsf(s[i]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  float amax = 0.0f;
#pragma unroll
  for (int w = 0; w < 8; ++w) amax = fmaxf(amax, red[w]);
  const float scale = fp8_scale(amax);
  if (threadIdx.x == 0) scales[blockIdx.x] = scale;
  for (int i = 2 * threadIdx.x; i < tileVals; i += 512) {
    const float lo = __fdiv_rn(s[i], scale);
    const float hi = (i + 1 < tileVals) ? __fdiv_rn(s[i + 1], scale) : 0.0f;
    const uint32_t two = fp8_two(lo, hi);
    d[i] = (uint8_t)(two & 0xffu);
    if (i + 1 < tileVals) d[i + 1] = (uint8_t)(two >> 8);
  }
}

template <int TPT>
void launch_fp8_tiles(const float* src, uint8_t* dst, float* scales, int nTiles, cudaStream_t s) {
  constexpr int tiles = kFp8Threads / TPT;
  k_to_fp8_tiles<TPT, 1><<<(nTiles + tiles - 1) / tiles, kFp8Threads, 0, s>>>(src, dst, scales,
                                                                             nTiles);
}

cudaError_t launch_fp8(const float* src, uint8_t* dst, float* scales, int nTiles, int tilePixels,
                       cudaStream_t s) {
  const bool aligned = ((uintptr_t)src | (uintptr_t)dst) % 16 == 0;
  switch (aligned ? tilePixels : 0) {
    case 16: launch_fp8_tiles<2>(src, dst, scales, nTiles, s); break;
    case 64: launch_fp8_tiles<8>(src, dst, scales, nTiles, s); break;
    case 256: launch_fp8_tiles<32>(src, dst, scales, nTiles, s); break;
    case 1024: launch_fp8_tiles<128>(src, dst, scales, nTiles, s); break;
    case 4096: launch_fp8_tiles<512>(src, dst, scales, nTiles, s); break;
    case 16384:
      if (nTiles <= 0x7fffffff / 4) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)nTiles * 4);
        cfg.blockDim = dim3(kFp8Threads);
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 4;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, k_to_fp8_tiles<4 * kFp8Threads, 4>, src, dst, scales,
                                  nTiles);
      }
      [[fallthrough]];
    default: k_to_fp8<<<nTiles, 256, 0, s>>>(src, dst, scales, tilePixels * 4);
  }
  return cudaGetLastError();
}

cudaError_t launch_convert(const float* src, void* dst, float* scales, int nTiles,
                           int tilePixels, int dtype, cudaStream_t s) {
  const int64_t n = (int64_t)nTiles * tilePixels * 4;
  switch (dtype) {
    case DFB_F16: launch_half(src, (__half*)dst, n, s); break;
    case DFB_BF16: launch_half(src, (__nv_bfloat16*)dst, n, s); break;
    case DFB_FP8E4M3: return launch_fp8(src, (uint8_t*)dst, scales, nTiles, tilePixels, s);
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace dfb
