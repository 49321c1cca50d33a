// dfb_composite_noalloc: one frame composited without allocating memory.
//
// Who needs this: callers that are not allowed to call cudaMalloc.  Examples
// are an in-situ simulation or renderer that reserves the whole device up
// front and hands out memory only from its own pool; real-time code where a
// cudaMalloc / cudaFree may synchronise the device and break a frame
// deadline; and code running where the CUDA runtime forbids allocation.  The
// handle-based path (dfb_create ... dfb_end_frame) allocates its framebuffers
// and bucketing scratch, so those callers cannot use it.
//
// This entry point keeps all its scratch (fragment records and the per-tile
// bucketing arrays) in one file-scope device array of fixed size, g_scratch,
// and writes only to the caller's output buffers.  It reuses the bucketing and
// composite kernels of the handle path unchanged.
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <memory>
#include <mutex>
#include <vector>

#include "dfb_internal.h"

namespace {

// Failure-detection settings of the calls (process-wide): the bound on every
// device-side wait, and a work item that the next call leaves unfilled.
std::atomic<unsigned long long> g_waitNs{2000000000ull};
std::atomic<int> g_stallItem{-1};

using dfb::FragRec;
using dfb::FrameArgs;

constexpr int kMaxFragments = 65536;  // fragment tiles per call
constexpr int kMaxTiles = 16384;      // tiles per frame
constexpr int kMaxRedo = 1 << 19;     // re-do units (32-pixel units of long tiles' items)

// Layout of g_scratch (each region 256-byte aligned):
//   stage: Header, then FragRec recs[n] (32 B each, grouped by tile) and int
//     tileOff[tiles + 1], as one upload of the call brings them
//   FragRec  srecs[kMaxFragments]     records sorted per tile
//   TileBlock blocks[kMaxTiles]       per-tile count/offset/first records
//   int      redo[kMaxRedo + 1]       the composite's re-do list
constexpr size_t align256(size_t v) { return (v + 255) & ~size_t(255); }
struct Header {
  dfb::FrameHeader frame;
  unsigned err;
};
constexpr size_t kHeaderBytes = align256(sizeof(Header));
constexpr size_t stage_bytes(size_t n, size_t tiles) {
  return kHeaderBytes + sizeof(FragRec) * n + sizeof(int) * (tiles + 1);
}
constexpr size_t kOffSrecs = align256(stage_bytes(kMaxFragments, kMaxTiles));
constexpr size_t kOffBlocks = align256(kOffSrecs + sizeof(FragRec) * kMaxFragments);
constexpr size_t kOffRedo = align256(kOffBlocks + sizeof(dfb::TileBlock) * kMaxTiles);
constexpr size_t kScratchBytes = align256(kOffRedo + sizeof(int) * (kMaxRedo + 1));  // ~15 MB

// The scratch itself.  Every GPU that loads the library holds it until the
// process exits.  In host code `g_scratch` names a host-side stand-in, not the
// device memory, so host code must only use the address that
// cudaGetSymbolAddress returns for the current device.
static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

// Device address of g_scratch per device, looked up once with that device
// current (the first call on a device does it).
std::mutex g_mu;
void* g_addr[64] = {};

int scratch_for_current_device(unsigned char** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return DFB_ERR_CUDA;
  std::lock_guard<std::mutex> lk(g_mu);
  if (!g_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess || !p) return DFB_ERR_CUDA;
    if (dfb::ensure_tables() != cudaSuccess) return DFB_ERR_CUDA;  // sRGB code boundaries
    g_addr[dev] = p;
  }
  *out = static_cast<unsigned char*>(g_addr[dev]);
  return DFB_OK;
}

bool device_accessible(const void* p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// Input tiles must be device (or managed) memory: the kernels read them with
// bulk copies.  Checking every pointer would cost one driver query per
// fragment tile, so only the first and the last tile of every run of
// back-to-back tiles (each starting `bytes` after the previous one, the
// layout of a pool) are checked.
template <class P>
bool tiles_accessible(const P* const* ptrs, int n, size_t bytes) {
  for (int i = 0; i < n;) {
    int j = i;
    while (j + 1 < n && reinterpret_cast<uintptr_t>(ptrs[j + 1]) ==
                            reinterpret_cast<uintptr_t>(ptrs[j]) + bytes)
      ++j;
    if (!device_accessible(ptrs[i]) || (j != i && !device_accessible(ptrs[j]))) return false;
    i = j + 1;
  }
  return true;
}

// The C entry point runs its body under this guard, so that no C++
// exception (a host vector that cannot grow) crosses the interface.
template <typename F>
int guarded_call(F&& body) noexcept {
  try {
    return body();
  } catch (const std::bad_alloc&) {
    return DFB_ERR_OOM;
  } catch (...) {
    return DFB_ERR_STATE;
  }
}

int composite_noalloc(int width, int height, int tile_size, int mode, int dtype, int n,
                      const int* tile_ids, const float* order_keys, const void* const* rgba,
                      const float* const* depth, const float* scales, const float* background,
                      float* color_out, uint32_t* rgba8_out, void* stream) {
  // ---- validation (host only) ----
  const int T = tile_size;
  if (width < 1 || height < 1 || T < 4 || T > 256 || (T & (T - 1))) return DFB_ERR_INVALID_ARG;
  if (mode < DFB_BLEND_DEPTH || mode > DFB_AVERAGE) return DFB_ERR_INVALID_ARG;
  if (dtype < DFB_F32 || dtype > DFB_FP8E4M3) return DFB_ERR_INVALID_ARG;
  if (n < 0 || (n > 0 && (!tile_ids || !order_keys || !rgba || !depth))) return DFB_ERR_INVALID_ARG;
  if (dtype == DFB_FP8E4M3 && n > 0 && !scales) return DFB_ERR_INVALID_ARG;
  if (!color_out && !rgba8_out) return DFB_ERR_INVALID_ARG;
  const int tilesX = (width + T - 1) / T, tilesY = (height + T - 1) / T;
  if ((int64_t)tilesX * tilesY > kMaxTiles || n > kMaxFragments) return DFB_ERR_CAPACITY;
  const int nTiles = tilesX * tilesY;
  // What the call uploads, in host memory: the header, the records grouped by
  // tile and the tiles' offsets.  Until the records are placed, off[t + 1]
  // counts tile t's.
  std::unique_ptr<unsigned char[]> stage(new unsigned char[stage_bytes((size_t)n, (size_t)nTiles)]);
  FragRec* const recs = reinterpret_cast<FragRec*>(stage.get() + kHeaderBytes);
  int* const off = reinterpret_cast<int*>(recs + n);
  std::fill(off, off + nTiles + 1, 0);
  int nLong = 0, nWindowed = 0;
  for (int i = 0; i < n; ++i) {
    if (tile_ids[i] < 0 || tile_ids[i] >= nTiles) return DFB_ERR_TILE_RANGE;
    const int c = ++off[tile_ids[i] + 1];
    if (c == dfb::kStageFragments + 1) ++nLong;
    if (c == dfb::kRedoRank + 1) ++nWindowed;
    if (isnan(order_keys[i]) || !rgba[i] || !depth[i]) return DFB_ERR_INVALID_ARG;
    if (((uintptr_t)rgba[i] % 16) || ((uintptr_t)depth[i] % 16)) return DFB_ERR_INVALID_ARG;
    if (dtype == DFB_FP8E4M3 && !(scales[i] > 0.0f && isfinite(scales[i])))
      return DFB_ERR_INVALID_ARG;
  }
  float bg[4] = {0.f, 0.f, 0.f, 0.f};
  if (background)
    for (int c = 0; c < 4; ++c) {
      if (!isfinite(background[c])) return DFB_ERR_INVALID_ARG;
      bg[c] = background[c];
    }
  cudaStream_t s = (cudaStream_t)stream;
  {
    // The call copies from pageable host memory and waits on the stream,
    // neither of which a capturing stream allows.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
      cudaGetLastError();
      return DFB_ERR_CUDA;
    }
    if (cap != cudaStreamCaptureStatusNone) return DFB_ERR_STATE;
  }
  if ((color_out && !device_accessible(color_out)) ||
      (rgba8_out && !device_accessible(rgba8_out)))
    return DFB_ERR_INVALID_ARG;
  const int chunksPerTile = T * T < dfb::kItemPixels ? 1 : T * T / dfb::kItemPixels;
  // only BLEND_DEPTH items of long tiles can need the re-do kernel
  const int64_t longItems = mode == DFB_BLEND_DEPTH ? (int64_t)nLong * chunksPerTile : 0;
  if (longItems * (dfb::kItemPixels / 32) > kMaxRedo) return DFB_ERR_CAPACITY;
  const size_t rgbaBytes = (size_t)T * T * 4 * (dtype == DFB_F32 ? 4 : (dtype == DFB_FP8E4M3 ? 1 : 2));
  if (!tiles_accessible(rgba, n, rgbaBytes) || !tiles_accessible(depth, n, (size_t)T * T * 4))
    return DFB_ERR_INVALID_ARG;

  unsigned char* base = nullptr;
  int st = scratch_for_current_device(&base);
  if (st != DFB_OK) return st;
  FragRec* srecs = reinterpret_cast<FragRec*>(base + kOffSrecs);
  dfb::TileBlock* blocks = reinterpret_cast<dfb::TileBlock*>(base + kOffBlocks);
  int* redo = reinterpret_cast<int*>(base + kOffRedo);
  Header* dHdr = reinterpret_cast<Header*>(base);
  dfb::LongList lng;
  if (longItems) {
    lng.windowed = nWindowed * (int)chunksPerTile;
    lng.ranked = (int)longItems - lng.windowed;
  }
  // each record at its place in the list grouped by tile (stable: submission
  // order kept within a tile)
  const bool fp8 = dtype == DFB_FP8E4M3;
  for (int t = 0; t < nTiles; ++t) off[t + 1] += off[t];
  {
    std::vector<int> cursor(off, off + nTiles);
    for (int i = 0; i < n; ++i) {
      FragRec& r = recs[cursor[tile_ids[i]]++];
      r.rgba = rgba[i];
      r.depth = depth[i];
      r.tile = (uint32_t)tile_ids[i];
      r.key = dfb::ordered_bits_host(order_keys[i]);
      r.scale = fp8 ? scales[i] : 1.0f;
      r.frame = 0u;
    }
  }

  Header& hdr = *reinterpret_cast<Header*>(stage.get());
  hdr = Header{};
  FrameArgs& a = hdr.frame.fa;
  dfb::frame_geometry(a, width, height, T);
  a.tileBase = 0;
  a.mode = mode;
  a.dtype = dtype;
  // no accumulation: the per-tile variance scratch of the handle path is unused
  a.flags = (color_out ? DFB_FLAG_WRITE_COLOR : 0u) | (rgba8_out ? DFB_FLAG_PACK_RGBA8 : 0u);
  a.frameN = 1;
  a.stateInRing = 0;  // no accumulation state
  a.keepTiles = dfb::kKeepAll;
  a.invN = 1.0f;
  a.invNm1 = 0.0f;
  a.bgR = bg[0] * bg[3];
  a.bgG = bg[1] * bg[3];
  a.bgB = bg[2] * bg[3];
  a.bgA = bg[3];
  a.pixelOp = DFB_PIXELOP_NONE;
  a.curve = nullptr;
  a.curveN = 0;
  a.curveXMax = 1.0f;
  a.curveScale = 0.0f;
  a.exposure = 1.0f;
  a.srecs = srecs;
  a.blocks = blocks;
  a.color = reinterpret_cast<float4*>(color_out);
  a.rgba8 = rgba8_out;
  int* const itemBase = hdr.frame.itemBase;
  itemBase[0] = 0;
  itemBase[1] = nTiles * a.chunks;
  hdr.err = 0u;

  // ---- one upload, bucketing (also clears the re-do count) and compositing.
  // The only wait is the one for the finished frame: the records are in this
  // call's own buffer, so the caller's arrays are free once it returns.
  // 1366x768, 4,333 fragment tiles: 91 us (114 us with an
  // upload per input array, waits between them and a packing kernel) ----
  cudaError_t e = cudaMemcpyAsync(base, stage.get(), stage_bytes((size_t)n, (size_t)nTiles),
                                  cudaMemcpyHostToDevice, s);
  const FragRec* dRecs = reinterpret_cast<const FragRec*>(base + kHeaderBytes);
  if (e == cudaSuccess)
    e = dfb::launch_bucket(dRecs, reinterpret_cast<const int*>(dRecs + n), nTiles, srecs, blocks,
                           redo, s);
  if (e != cudaSuccess) {
    cudaStreamSynchronize(s);  // the upload has left the host buffer
    return e == cudaErrorMemoryAllocation ? DFB_ERR_OOM : DFB_ERR_CUDA;
  }
  const dfb::LaunchCtl ctl{g_waitNs.load(), g_stallItem.exchange(-1), &dHdr->err, redo};
  e = dfb::launch_composite(&dHdr->frame.fa, dHdr->frame.itemBase, 1, itemBase[1], nTiles, false,
                           dtype,
                           dfb::default_tune(dtype, (double)n / (double)nTiles, true), ctl, lng,
                           &a, itemBase, nullptr, s);
  if (e != cudaSuccess) {
    cudaStreamSynchronize(s);  // the upload has left the host buffer
    return DFB_ERR_CUDA;
  }
  // The launch's error word: a wait that ran out (the frame is then
  // incomplete) or, in the checked build, a failed device-side check.  The
  // next call clears it, so it is read here, once the frame is done.
  unsigned err = 0u;
  e = cudaMemcpyAsync(&err, &dHdr->err, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return DFB_ERR_CUDA;
  if (err & dfb::kErrCheck) return DFB_ERR_CHECK;
  if (err) return DFB_ERR_TIMEOUT;
  return DFB_OK;
}

}  // namespace

extern "C" int dfb_noalloc_set_wait_limit(double seconds) {
  if (!(seconds > 0.0) || seconds > 3600.0) return DFB_ERR_INVALID_ARG;
  g_waitNs.store((unsigned long long)(seconds * 1e9));
  return DFB_OK;
}

extern "C" int dfb_noalloc_inject_stall(int item) {
  if (item < -1) return DFB_ERR_INVALID_ARG;
  g_stallItem.store(item);
  return DFB_OK;
}

extern "C" int dfb_composite_noalloc(int width, int height, int tile_size, int mode, int dtype,
                                     int n, const int* tile_ids, const float* order_keys,
                                     const void* const* rgba, const float* const* depth,
                                     const float* scales, const float* background,
                                     float* color_out, uint32_t* rgba8_out, void* stream) {
  return guarded_call([&]() -> int {
    return composite_noalloc(width, height, tile_size, mode, dtype, n, tile_ids, order_keys, rgba,
                             depth, scales, background, color_out, rgba8_out, stream);
  });
}
