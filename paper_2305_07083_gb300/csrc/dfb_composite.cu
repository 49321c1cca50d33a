// Composite kernel of the DFB path (K2/K3 with the fused K4 epilogue) for
// sm_103a: a persistent, warp-specialised, bulk-copy pipeline.
//
// Per pixel it computes the AlphaBlend tile operation of Sec. 4.2 /
// Listing 4 (sort the pixel's fragments by depth -- ties by order key, then
// submit index -- and blend them front to back with the premultiplied "over"
// operator, then the generation-0 background of Listing 3), the ordered
// "list" form of Sec. 4.2 (blend in key order), depth compositing (Sec. 2.1:
// the nearest fragment's RGBA), or the mean of redundantly rendered tiles
// (Sec. 4.1.1), and an optional pixel operation before the display
// conversion (Sec. 3.1.2).  The epilogue updates the
// progressive accumulation and variance tiles of Listing 1 (running sum,
// Kahan-compensated past a threshold; Welford M2; per-tile variance for
// Sec. 4.1.1) and writes the RGBA8 display format of Sec. 3.1.
//
// The work is bound by HBM bandwidth (~0.4 flop per byte), so the design goal
// is to keep enough bytes in flight:
//   * CTA = G consumer groups of 8 warps (one pixel per thread, 256 pixels =
//     one work item; the groups take alternate items) + 1 producer warp, PER
//     CTAs per SM (by default G = 1 and PER = 2 or 3, by default_tune).
//     CTAs are persistent and walk the work items of all frames of the launch
//     with a static stride, which keeps the chunks of a tile on neighbouring
//     CTAs that run in step.
//   * The producer warp takes its items in rounds of kRound.  It fetches a
//     round's tile blocks (fragment count, list offset and sorted records,
//     written by the bucketing) two rounds ahead, a bulk copy each and one
//     barrier for all, so locating an item's fragments needs no dependent
//     global loads.  It then issues one-dimensional bulk copies
//     (cp.async.bulk, the TMA engine) of each fragment's depth slab and RGBA
//     slab straight into a shared-memory ring, completing on the fill's
//     mbarrier.  Fills take only the ring bytes they need (n fragments x slab
//     size), so the ring holds as many fills in flight as their sizes allow,
//     up to kSlots (each consumer group owns kSlots / G of them).
//   * An item of at most kStageFragments fragments is one fill.  A longer
//     one streams through the ring in fills of kFill fragments; its
//     consumers carry the per-pixel blend across the fills (BLEND_DEPTH
//     speculatively in list order), so a long list costs the same bytes per
//     fragment as a short one.  The rare 32-pixel units whose depths turn
//     out to be out of list order are redone exactly by k_composite_redo.
//   * The accumulation state (sum, M2, Kahan compensation) is stored
//     tile-major, so an item's state is one contiguous run per buffer.  In
//     frames with few fragments per tile the producer streams it into the
//     item's last fill; in the others the consumers load it into registers
//     before they wait for the fragments, so that the ring holds fragments
//     only (the state's bytes would occupy it for the item's whole stay and
//     leave room for fewer items in flight).  Consumers read the fragments
//     from shared memory, sort and blend, and release the ring space before
//     the epilogue.
//   * The epilogue writes one variance partial per warp with plain stores;
//     a small second kernel sums each tile's partials in a fixed order.
// Every wait is bounded in time; on expiry the kernel sets an error bit,
// drains its own bulk copies and returns.
#include <string.h>

#include "dfb_device.cuh"
#include "dfb_internal.h"

namespace dfb {

// sRGB encode tables (SrgbTables), uploaded by the host.
__device__ SrgbTables g_srgb;

cudaError_t upload_srgb_tables(const SrgbTables& host) {
  return cudaMemcpyToSymbol(g_srgb, &host, sizeof(SrgbTables));
}

// Copy the sRGB tables into shared memory (every thread of the CTA calls it).
__device__ __forceinline__ void load_srgb(SrgbTables* dst, int nThreads) {
  const uint32_t* src = reinterpret_cast<const uint32_t*>(&g_srgb);
  uint32_t* d = reinterpret_cast<uint32_t*>(dst);
  for (int i = threadIdx.x; i < (int)(sizeof(SrgbTables) / 4); i += nThreads) d[i] = src[i];
}

namespace {

constexpr int kP = kItemPixels;          // pixels per item = threads of a consumer group
constexpr int kCW = kP / 32;             // warps of a consumer group
// Threads of a CTA with G consumer groups (items k, k+1, ... composited in
// parallel) and one producer warp.
template <int G>
struct Shape {
  static constexpr int threads = G * kP + 32;
  static_assert(threads <= 1024, "threads per CTA");
};
// Launch shapes: G consumer groups per CTA, PER resident CTAs per SM.
//   (G, PER) = (1, 2), (2, 2), (1, 3), (2, 1), (3, 1)
constexpr int kN = kStageFragments;
constexpr int kSlots = 16;               // items in flight at most
constexpr int kRound = 4;                // items the producer plans at once
constexpr int kMetaQ = 2 * kRound;       // tile blocks fetched ahead
constexpr uint32_t kWindowBytes = kSortWindow * kP * 8;
constexpr int kRedoPer = 3;              // CTAs per SM of the re-do, by ranks
constexpr int kWindowPer = 3;            // and by windowed rounds

// Descriptor of one fill of the ring: up to kN fragments of one work item
// (all of them for an item of at most kN fragments, else kFill), and the
// item's state rows in its last fill when the frame streams them.
struct __align__(16) ItemMeta {
  int n;               // fragments in this fill
  int total;           // fragments of the item
  int pad0;            // n to start are one 16-byte store, bytes and end one of 8
  uint32_t start;      // byte offset of the fill's data in the ring
  uint32_t bytes;      // bytes of the fill's fragments from `start` (state rows follow)
  uint32_t end;        // producer's head count after this fill (modulo 2^32)
  uint32_t pad[2];
  const void* rgba[kN];  // ZCOMPOSITE: the fragments' RGBA in global memory
  float scale[kN];       // FP8: the fragments' scales
};
static_assert(sizeof(ItemMeta) <= 256, "item meta");

// Shared memory: [sRGB tables 2.75 KB][barriers 512 B][flags 128 B][metas 4 KB]
//                [tile-block queue][ring]
constexpr int kOffBars = (int)sizeof(SrgbTables);
constexpr int kOffFlags = kOffBars + 512;
constexpr int kOffMetas = kOffFlags + 128;
constexpr int kOffQueue = kOffMetas + kSlots * 256;
constexpr int kHeader = kOffQueue + kMetaQ * (int)sizeof(TileBlock);
static_assert((2 * kSlots + 2) * 8 <= 512, "barrier space");
static_assert(kOffQueue % 128 == 0 && kHeader % 128 == 0, "alignment");
static_assert(32 % kFill == 0 && kFill <= kN, "fills never straddle a window of 32 records");

template <int DT>
struct Bytes {
  static constexpr int px = PxBytes<DT>::value;
  // largest fill the ring must hold: kN fragments plus three rows of
  // framebuffer state (sum, M2, Kahan compensation)
  static constexpr uint32_t maxItem = (uint32_t)kN * kP * (4 + px) + 3u * kP * 16u;
};

// Where a launch's frame arguments are read from.
constexpr int kGlobalTable = 0;  // the frame table and item prefix in global memory
constexpr int kOneFrame = 1;     // one frame, its arguments a kernel parameter
constexpr int kParamTable = 2;   // up to kParamFrames frames, the tables a kernel parameter
constexpr int kParamFrames = 48;
struct FrameTable {
  int itemBase[kParamFrames + 1];
  FrameArgs f[kParamFrames];
};
static_assert(sizeof(FrameTable) <= 16384, "kernel parameter size");
// Whether a launch's frames choose what stays in L2 (FrameArgs::keepTiles).
template <int FR>
constexpr bool kKeeps = FR == kOneFrame;
template <int FR>
struct FrameParams {
  using type = int;  // unused
};
template <>
struct FrameParams<kOneFrame> {
  using type = FrameArgs;
};
template <>
struct FrameParams<kParamTable> {
  using type = FrameTable;
};

__device__ __forceinline__ int find_frame(const int* itemBase, int nFrames, int item) {
  int lo = 0, hi = nFrames - 1;  // last frame whose first item <= item
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (itemBase[mid] <= item) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Bounded wait on an mbarrier phase.  Returns false when the wait expired or
// another role of the CTA has given up.
__device__ __forceinline__ bool wait_phase(uint64_t* bar, uint32_t parity, const LaunchCtl& ctl,
                                           volatile int* abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  for (uint32_t spin = 1;; ++spin) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((spin & 63) == 0) {
      if (*abort) return false;
      if (global_ns() - t0 > ctl.waitNs) return false;
    }
  }
}

__device__ __forceinline__ void give_up(const LaunchCtl& ctl, volatile int* abort) {
  *abort = 1;
  atomicOr(ctl.err, kErrTimeout);
}

// Insert k into the sorted per-thread window kb[0..m-1] (stride kP),
// shifting larger keys up one slot; slot m must be free.
__device__ __forceinline__ void window_insert(uint64_t* kb, int m, uint64_t k) {
  int j = m - 1;
  while (j >= 0) {
    const uint64_t v = kb[j * kP];
    if (v < k) break;
    kb[(j + 1) * kP] = v;
    --j;
  }
  kb[(j + 1) * kP] = k;
}

// The frame of work item `item`, given the frame `f` of an earlier one: a
// role's items only ascend, so the search is a step at most frames' ends.
// FR: where the launch's frame arguments are (FrameSource); with kOneFrame
// `frames` points to a single frame's arguments in the kernel's parameter
// space (read through the constant cache, no loads).
template <int FR>
__device__ __forceinline__ int next_frame(const int* itemBase, int f, int item) {
  if (FR != kOneFrame)
    while (item >= itemBase[f + 1]) ++f;
  return f;
}

// ---------------------------------------------------------------------------
// producer warp
// ---------------------------------------------------------------------------
// Fills of the ring.  Consumer group g owns the slots g*S .. g*S+S-1 (S =
// kSlots / G) and takes its items' fills from them in order.  Ring bytes are
// reclaimed in the global order of the fills; a fill may reuse a slot once
// the slot's previous fill has been released.
//
// One warp feeds the CTA, and with slabs of 1 to 4 KB its own time per item
// sets the pace long before the ring is full, so that time is kept short:
//   * the items are planned kRound at a time, a lane per item (frame, tile,
//     sizes, the fetch of its tile block), one wait per round;
//   * ring positions are 32-bit counters and an offset, with no division;
//   * an item's descriptor is two 16-byte stores, and pointers and scales
//     are stored only for the modes and formats that read them.
// Measured, FP16, mixed frames in one launch (2 CTAs per SM): 3,300 cycles of
// this warp per item before, of which it waited for space in none; the launch
// of 16 frames 1.013 -> 0.708 ms, a server's step of 8 frames of one fragment
// per tile 0.219 -> 0.184 ms.
template <int DT, int G, int FR>
__device__ void producer(const FrameArgs* __restrict__ frames, const int* __restrict__ itemBase,
                         int nFrames, int totalItems, const LaunchCtl& ctl, unsigned char* ring,
                         uint32_t ringBytes, ItemMeta* metas, TileBlock* queue, uint64_t* fullB,
                         uint64_t* emptyB, uint64_t* queueB, volatile int* abort) {
  constexpr int px = Bytes<DT>::px;
  constexpr int S = kSlots / G;
  const int lane = threadIdx.x & 31;
  // Ring bytes handed out and reclaimed since the start, modulo 2^32 (their
  // difference is what is outstanding), and the offset of the next fill.
  uint32_t head = 0, tail = 0, pos = 0;
  int curFill = 0, tailFill = 0;          // fills issued / reclaimed (global order)
  int gf0 = 0, gf1 = 0, gf2 = 0;          // fills issued per consumer group
  // With one group, fill e lies in slot e mod kSlots.  With several, lane e <
  // kSlots holds the slot and the parity of outstanding fill e (mod kSlots)
  // and lane s < kSlots the global index of the last fill of slot s.
  int fifoSlot = 0, fifoPar = 0, slotFill = -1;
  uint32_t armed = 0, armedPar = 0;       // per ring slot: armed / parity of last arm
  uint32_t qArmed = 0, qPar = 0;          // per half of the tile-block queue
  // Bytes of one fragment's slabs and rows of state of a frame's items: the
  // depth slab | the RGBA slab << 16, and the pixels per item | state rows <<
  // 16 | winner only (ZCOMPOSITE) << 24.
  struct Sizes {
    uint32_t bytes, more;
  };
  auto sizes = [](const FrameArgs* A) -> Sizes {
    const int P = A->P, mode = A->mode;
    const uint32_t dBytes =
        mode == DFB_BLEND_DEPTH || mode == DFB_ZCOMPOSITE ? (uint32_t)P * 4u : 0u;
    const uint32_t cBytes = mode != DFB_ZCOMPOSITE ? (uint32_t)P * px : 0u;
    // accumulation state of the item's pixels, one contiguous run per
    // buffer, when the frame streams it with the fragments
    const bool loadState = (A->flags & DFB_FLAG_ACCUMULATE) && A->frameN != 1 && A->stateInRing;
    const int nState = loadState ? (A->kahan && !A->kahanFirst ? 3 : 2) : 0;
    return Sizes{dBytes | cBytes << 16, (uint32_t)P | (uint32_t)nState << 16 |
                                            (mode == DFB_ZCOMPOSITE ? 1u << 24 : 0u)};
  };
  // Round r's plan: lane u < kRound has item r * kRound + u of this CTA.  In
  // a single-frame launch the sizes are the frame's.
  struct Plan {
    int f, tile, chunk;
    Sizes sz;
  };
  const Sizes one = FR == kOneFrame ? sizes(frames) : Sizes{};
  const uint64_t evictFirst = l2_evict_first();
  int scanF = 0;
  auto plan = [&](int r) -> Plan {
    Plan p{};
    const int it = blockIdx.x + (r * kRound + lane) * (int)gridDim.x;
    const bool valid = lane < kRound && it < totalItems;
    const int count = __popc(__ballot_sync(0xffffffffu, valid));
    if (count == 0) return p;
    const int half = r & 1;
    int gt = 0;
    if (valid) {
      scanF = next_frame<FR>(itemBase, scanF, it);
      const FrameArgs* A = frames + (FR == kOneFrame ? 0 : scanF);
      const int local = FR == kOneFrame ? it : it - itemBase[scanF];
      p.f = scanF;
      p.tile = local >> A->logChunks;
      p.chunk = local & (A->chunks - 1);
      gt = A->tileBase + p.tile;
      if (FR != kOneFrame) p.sz = sizes(A);
    }
    const bool fits = DFB_CHECK(!valid || (p.f < nFrames && p.tile < frames[p.f].nTiles), ctl.err);
    // the slots' previous blocks were read through the generic proxy
    fence_proxy_async();
    if (lane == 0) mbar_arrive_expect_tx(&queueB[half], (uint32_t)count * (uint32_t)sizeof(TileBlock));
    __syncwarp();
    if (valid)
      bulk_g2s(queue + half * kRound + lane, frames[p.f].blocks + (fits ? gt : 0),
               (uint32_t)sizeof(TileBlock), &queueB[half]);
    qArmed |= 1u << half;
    qPar = (qPar & ~(1u << half)) | ((uint32_t)((r >> 1) & 1) << half);
    return p;
  };
  Plan cur = plan(0), next = plan(1);
  bool ok = true;
  for (int r = 0;; ++r) {
    const int k0 = r * kRound;
    if (blockIdx.x + (long long)k0 * gridDim.x >= totalItems) break;
    const int half = r & 1;
    if (!wait_phase(&queueB[half], (uint32_t)(r >> 1) & 1u, ctl, abort)) {
      ok = false;
      break;
    }
    // The round's tile blocks stay in their half of the queue until its
    // fills are issued; the fetch of the round after the next follows them.
    const int myN = lane < kRound ? queue[half * kRound + lane].n : 0;
    for (int u = 0; u < kRound && ok; ++u) {
      const int k = k0 + u;
      const int item = blockIdx.x + k * (int)gridDim.x;
      if (item >= totalItems) break;
      const TileBlock* blk = queue + half * kRound + u;
      const int n = __shfl_sync(0xffffffffu, myN, u);
      const FrameArgs* A = frames + (FR == kOneFrame ? 0 : __shfl_sync(0xffffffffu, cur.f, u));
      const uint32_t bytes =
          FR == kOneFrame ? one.bytes : __shfl_sync(0xffffffffu, cur.sz.bytes, u);
      const uint32_t more = FR == kOneFrame ? one.more : __shfl_sync(0xffffffffu, cur.sz.more, u);
      const int chunk =
          FR == kOneFrame ? item & (A->chunks - 1) : __shfl_sync(0xffffffffu, cur.chunk, u);
      const uint32_t cBytes = bytes >> 16;
      // a single fragment to blend needs no depth (item_mode)
      const uint32_t dBytes = n == 1 && cBytes ? 0u : bytes & 0xffffu;
      const int P = (int)(more & 0xffffu), nState = (int)(more >> 16 & 0xffu);
      const size_t p0 = (size_t)chunk * P;  // the item's first pixel in its tile
      // An item of more than kN fragments is streamed in fills of kFill; its
      // records past the tile block come from the sorted list.
      const int per = n > kN ? kFill : kN;
      const int fills = n > kN ? (n + kFill - 1) / kFill : 1;
      const int g = G == 1 ? 0 : k % G;
      for (int f = 0; f < fills; ++f) {
        const int i0 = f * per;
        const int nf = min(per, n - i0);
        const bool lastFill = f == fills - 1;
        const uint32_t fragBytes = (uint32_t)nf * (dBytes + cBytes);
        const uint32_t need =
            fragBytes + (lastFill ? nState * (uint32_t)P * 16u : 0u);  // multiple of 16
        // lane li < nf takes fragment i0 + li: from the tile block for the
        // first kN, else from the sorted list in global memory
        const void* rRgba = nullptr;
        const float* rDepth = nullptr;
        float rScale = 1.0f;
        if (lane < nf) {
          const int i = i0 + lane;
          if (i < kN) {
            rRgba = blk->recs[i].rgba;
            rDepth = blk->recs[i].depth;
            if (DT == DFB_FP8E4M3) rScale = blk->recs[i].scale;
          } else {
            const FragRec* rec = A->srecs + blk->off + i;
            rRgba = rec->rgba;
            rDepth = rec->depth;
            if (DT == DFB_FP8E4M3) rScale = rec->scale;
          }
        }
        // ring space: no fill straddles the end of the ring
        if (pos + need > ringBytes) {
          head += ringBytes - pos;
          pos = 0;
        }
        // everything but the stores and copies themselves is ready before the
        // wait for space, so that freed space is refilled at once
        const uint32_t start = pos;
        const float* dSrc = rDepth + p0;
        const unsigned char* cSrc = static_cast<const unsigned char*>(rRgba) + p0 * px;
        unsigned char* dDst = ring + start + lane * dBytes;
        unsigned char* cDst = ring + start + nf * dBytes + lane * cBytes;
        const int jg = G == 1 ? curFill : (g == 0 ? gf0 : (g == 1 ? gf1 : gf2));
        const int s = g * S + jg % S;
        const uint32_t par = (uint32_t)(jg / S) & 1u;
        const int prev =
            G == 1 ? curFill - kSlots : __shfl_sync(0xffffffffu, slotFill, s);
        while (tailFill < curFill && (tailFill <= prev || head + need - tail > ringBytes)) {
          const int e = tailFill % kSlots;
          const int es = G == 1 ? e : __shfl_sync(0xffffffffu, fifoSlot, e);
          const int ep =
              G == 1 ? (tailFill / kSlots) & 1 : __shfl_sync(0xffffffffu, fifoPar, e);
          if (!wait_phase(&emptyB[es], (uint32_t)ep, ctl, abort)) {
            ok = false;
            break;
          }
          tail = metas[es].end;
          ++tailFill;
        }
        if (!ok) break;
        if (tailFill == curFill) tail = head;  // nothing outstanding: the padding is free too
        if (!DFB_CHECK(pos + need <= ringBytes && head + need - tail <= ringBytes && nf <= kN &&
                           (chunk + 1) * P <= A->T * A->T,
                       ctl.err)) {
          ok = false;
          break;
        }
        head += need;
        pos += need;
        ItemMeta* meta = metas + s;
        if (lane < nf) {
          if (more >> 24) meta->rgba[lane] = rRgba;
          if (DT == DFB_FP8E4M3) meta->scale[lane] = rScale;
        }
        if (lane == 0) {
          *reinterpret_cast<int4*>(&meta->n) = make_int4(nf, n, 0, (int)start);
          *reinterpret_cast<uint2*>(&meta->bytes) = make_uint2(fragBytes, head);
        }
        if (G > 1) {
          if (lane == curFill % kSlots) {
            fifoSlot = s;
            fifoPar = (int)par;
          }
          if (lane == s) slotFill = curFill;
          if (g == 0) ++gf0; else if (g == 1) ++gf1; else ++gf2;
        }
        ++curFill;
        __syncwarp();
        if (f != 0 || item != ctl.stallItem) {  // test fault injection: never signal this item
          if (lane == 0) mbar_arrive_expect_tx(&fullB[s], need);
          armed |= 1u << s;
          armedPar = (armedPar & ~(1u << s)) | (par << s);
          __syncwarp();
          if (kKeeps<FR> && A->keepTiles != kKeepAll) {
            if (lane < nf) {
              if (dBytes) bulk_g2s_hint(dDst, dSrc, dBytes, &fullB[s], evictFirst);
              if (cBytes) bulk_g2s_hint(cDst, cSrc, cBytes, &fullB[s], evictFirst);
            }
          } else if (lane < nf) {
            if (dBytes) bulk_g2s(dDst, dSrc, dBytes, &fullB[s]);
            if (cBytes) bulk_g2s(cDst, cSrc, cBytes, &fullB[s]);
          }
          if (lastFill && nState) {
            // state runs: [sum | M2 | comp], P pixels of 16 bytes each
            const int tile =
                FR == kOneFrame ? item >> A->logChunks : __shfl_sync(0xffffffffu, cur.tile, u);
            if (lane < nState) {
              const float4* src = lane == 0 ? A->accum : (lane == 1 ? A->m2 : A->comp);
              void* dst = ring + start + fragBytes + lane * (uint32_t)P * 16u;
              src += (size_t)tile * A->T * A->T + p0;
              if (kKeeps<FR> && tile >= A->keepTiles)
                bulk_g2s_hint(dst, src, (uint32_t)P * 16u, &fullB[s], evictFirst);
              else
                bulk_g2s(dst, src, (uint32_t)P * 16u, &fullB[s]);
            }
          }
        }
      }
    }
    if (!ok) break;
    __syncwarp();  // every lane is done with the half's blocks
    cur = next;
    next = plan(r + 2);
  }
  if (!ok && lane == 0) give_up(ctl, abort);
  // Leave no bulk copy in flight into this CTA's shared memory.
  auto drain = [&](uint64_t* bars, uint32_t mask, uint32_t parv, int count) {
    for (int qq = 0; qq < count; ++qq)
      if (mask & (1u << qq)) {
        const uint64_t t0 = global_ns();
        while (!mbar_try_wait(&bars[qq], (parv >> qq) & 1u)) {
          if (global_ns() - t0 > ctl.waitNs) {
            if (lane == 0) atomicOr(ctl.err, kErrDrain);
            break;
          }
        }
      }
  };
  drain(fullB, armed, armedPar, kSlots);
  drain(queueB, qArmed, qPar, 2);
}

// ---------------------------------------------------------------------------
// consumer warps: one pixel per thread
// ---------------------------------------------------------------------------
// A depth that takes part in the blend: not +inf and not NaN (both read as an
// empty fragment; NaN maps to +inf).  The speculative in-order passes compare
// such depths as floats, which orders them exactly as their canonical keys
// (depth_bits) do: -0 equals +0 and -inf comes first.
__device__ __forceinline__ bool covers(float z) { return z <= 3.402823466e38f; }

// One fill's `n` fragments at pixel t of the item, in list order, behind what
// is accumulated: the speculative pass of BLEND_DEPTH.  For bricks whose key
// order is their depth order (the common case) the finite-depth fragments
// are already in blend order, so they are blended as they are read while the
// order is checked.  A fragment empty at this pixel (depth +inf or NaN, which
// sorts after every finite depth) is blended with weight zero: an all-zero
// RGBA is an exact no-op anywhere in the order.  `last` is the last finite
// depth, `bad` says that the depths were out of order, `rest` collects the
// bits of the empty fragments' RGBA.  The result stands if neither is set;
// else the caller blends the empty ones behind it, or starts the pixel over
// in exact order.
//
// The loop body has no branch (the weight, the order check and the bits are
// selects), so that the shared-memory loads of four fragments are in flight
// at once.  P is the constant kP in all but the smallest tiles (FULL): the
// slabs' addresses are then one register plus constants.  16-frame
// accumulation at 2048x2048 in FP16: 1.764 -> 1.739 ms; 1024x1024 with
// overlapping producers, FP32: 117.8 -> 113.8 us.
template <int DT, bool FULL>
__device__ __forceinline__ void blend_in_order(int n, int stride, const unsigned char* base,
                                               const ItemMeta* meta, int t, float& c0, float& c1,
                                               float& c2, float& al, float& last, bool& bad,
                                               uint32_t& rest) {
  constexpr int px = Bytes<DT>::px;
  const int P = FULL ? kP : stride;
  const float* sD = reinterpret_cast<const float*>(base) + t;
  const unsigned char* sC = base + (size_t)n * P * 4;
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    const float z = sD[i * P];
    const typename Px<DT>::Raw v = Px<DT>::raw(sC + (size_t)i * P * px, t);
    const float4 f = Px<DT>::decode(v, DT == DFB_FP8E4M3 ? meta->scale[i] : 1.0f);
    const bool in = covers(z);
    const float w = in ? 1.0f - al : 0.0f;
    c0 = fmaf(w, f.x, c0);
    c1 = fmaf(w, f.y, c1);
    c2 = fmaf(w, f.z, c2);
    al = fmaf(w, f.w, al);
    const float zz = in ? z : last;
    bad = bad || zz < last;
    last = zz;
    rest |= in ? 0u : Px<DT>::bits(v);
  }
}

// The mode by which an item of `n` fragments is composited: a single fragment
// has no order, so BLEND_DEPTH does not read its depth (an empty one is
// blended too, as the last).  A server's step of 8 frames of one fragment per
// tile, FP16, accumulating: launch 184.5 -> 176.7 us.
__device__ __forceinline__ int item_mode(int mode, int n) {
  return mode == DFB_BLEND_DEPTH && n == 1 ? (int)DFB_BLEND_ORDERED : mode;
}

// The nearest of one fill's `n` fragments at pixel t against `z`, the nearest
// depth so far: its index in the fill, or -1.  The first of equal depths stays
// (list order); +inf and NaN are no fragment.  No branch and no 64-bit key:
// launch of 1920x1080, BF16, 3.5 fragments per tile: 43.2 -> 41.4 us.
template <bool FULL>
__device__ __forceinline__ int nearest(int n, int stride, const float* sD, int t, float& z) {
  const int P = FULL ? kP : stride;
  int best = -1;
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    const float v = sD[i * P + t];
    best = v < z ? i : best;  // false for a NaN
    z = v < z ? v : z;
  }
  return best;
}

// One fill's `n` fragments behind what is accumulated, in list order: all of
// them (BLEND_ORDERED), or added up (AVERAGE).
template <int DT, int MODE, bool FULL>
__device__ __forceinline__ void blend_list(int n, int stride, const unsigned char* sC,
                                           const ItemMeta* meta, int t, float& c0, float& c1,
                                           float& c2, float& al) {
  constexpr int px = Bytes<DT>::px;
  const int P = FULL ? kP : stride;
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    const float4 f =
        Px<DT>::shared(sC + (size_t)i * P * px, t, DT == DFB_FP8E4M3 ? meta->scale[i] : 1.0f);
    if (MODE == DFB_BLEND_ORDERED) {
      over(f, c0, c1, c2, al);
    } else {
      c0 += f.x; c1 += f.y; c2 += f.z; al += f.w;
    }
  }
}

// Returns false only in DFB_ZCOMPOSITE for a pixel no fragment covers.
template <int DT, bool FULL>
__device__ __forceinline__ bool composite_staged(int mode, int n, int P, const unsigned char* base,
                                                 const ItemMeta* meta, int t, int p,
                                                 float& c0, float& c1, float& c2, float& al) {
  constexpr int px = Bytes<DT>::px;
  const float* sD = reinterpret_cast<const float*>(base);
  // floats per depth slab (no depth is staged in the modes that ignore it)
  const int dStride = mode == DFB_BLEND_DEPTH || mode == DFB_ZCOMPOSITE ? P : 0;
  const unsigned char* sC = base + (size_t)n * dStride * 4;
  const int stride = FULL ? kP : P;
  if (mode == DFB_BLEND_ORDERED) {
    blend_list<DT, DFB_BLEND_ORDERED, FULL>(n, P, sC, meta, t, c0, c1, c2, al);
  } else if (mode == DFB_AVERAGE) {
    // equal-weight mean of the redundant tiles, summed in list order
    blend_list<DT, DFB_AVERAGE, FULL>(n, P, sC, meta, t, c0, c1, c2, al);
    if (n > 0) {
      const float k = (float)n;
      c0 = __fdiv_rn(c0, k); c1 = __fdiv_rn(c1, k); c2 = __fdiv_rn(c2, k); al = __fdiv_rn(al, k);
    }
  } else if (mode == DFB_ZCOMPOSITE) {
    float z = INFINITY;
    const int i = nearest<FULL>(n, P, sD, t, z);
    if (i < 0) return false;
    const float4 f = Px<DT>::global(meta->rgba[i], p, meta->scale[i]);
    c0 = f.x; c1 = f.y; c2 = f.z; al = f.w;
  } else {
    {
      float last = -INFINITY;
      uint32_t rest = 0;
      bool bad = false;
      blend_in_order<DT, FULL>(n, P, base, meta, t, c0, c1, c2, al, last, bad, rest);
      if (!bad && rest == 0u) return true;
      // In order, but empty fragments carry colour (renderers that write no
      // depth): what is blended stands, and they follow in list order.  Only
      // an infinity or NaN of theirs can have spoilt it (0 times it is NaN,
      // and NaN stays).  1024x1024 FP32, 16 fragments per tile without
      // depths: 99 us with a sort instead, 87 so; 2048x1024 FP16, 8 per tile:
      // 99 and 82.
      if (!bad && !isnan(c0 + c1 + c2 + al)) {
#pragma unroll 1
        for (int i = 0; i < n; ++i)
          if (!covers(sD[i * stride + t]))
            over(Px<DT>::shared(sC + (size_t)i * P * px, t, meta->scale[i]), c0, c1, c2, al);
        return true;
      }
      c0 = c1 = c2 = al = 0.0f;
    }
    // General case: sort of fragment indices (4-bit slots of `perm`) by
    // depth.  The list arrives in key order, so ties stay in (key, submit
    // index) order; empty fragments go to a second list kept in list order
    // and blended last.  A finite fragment goes in front of the finite ones
    // before it that are deeper: all deeper depths in the list so far are
    // counted, by loads that do not depend on one another, and the infinite
    // ones (`far`) taken off.  Two fragments share the loads, and a pair that
    // is at least as deep as all before it needs no count, so that a list
    // nearly in order costs little.  2048x1024 FP16, 16 fragments of which two
    // are swapped, 174 us, 244 with a count for every fragment by itself;
    // random order, 1024x1024 FP32, 123 and 131 (by insertion 176 and 252).
    const float* zt = sD + t;
    uint64_t perm = 0, infs = 0;
    int m = 0, mi = 0, far = 0;
    float deepest = -INFINITY;
    auto place = [&](int i, bool in, int deeper) {
      const int at = 4 * (m - (in ? deeper : 0));
      const uint64_t low = perm & ((1ull << at) - 1ull);
      const uint64_t put = low | ((uint64_t)i << at) | ((perm ^ low) << 4);
      perm = in ? put : perm;
      infs |= in ? 0ull : (uint64_t)i << (4 * mi);
      m += in ? 1 : 0;
      mi += in ? 0 : 1;
    };
    for (int i = 0; i < n; i += 2) {
      const bool two = i + 1 < n;
      const float z0 = zt[i * stride];
      const float z1 = two ? zt[(i + 1) * stride] : NAN;
      const bool in0 = covers(z0), in1 = covers(z1);
      const float mid = in0 ? fmaxf(deepest, z0) : deepest;
      int d0 = 0, d1 = 0;
      if ((in0 && z0 < deepest) || (in1 && z1 < mid)) {
        d0 = -far;
        d1 = in0 && z0 > z1 ? 1 - far : -far;
#pragma unroll 2
        for (int j = 0; j < i; ++j) {
          const float v = zt[j * stride];
          d0 += v > z0 ? 1 : 0;
          d1 += v > z1 ? 1 : 0;
        }
      }
      place(i, in0, d0);
      if (two) place(i + 1, in1, d1);
      deepest = in1 ? fmaxf(mid, z1) : mid;
      far += (z0 == INFINITY ? 1 : 0) + (z1 == INFINITY ? 1 : 0);
    }
    // one loop of exactly n steps: the finite list, then the empty ones
#pragma unroll 2
    for (int r = 0; r < n; ++r) {
      const bool fin = r < m;
      const uint64_t src = fin ? perm : infs;
      const int rr = fin ? r : r - m;
      const int i = (int)((src >> (4 * rr)) & 15u);
      over(Px<DT>::shared(sC + (size_t)i * P * px, t, meta->scale[i]), c0, c1, c2, al);
    }
  }
  return true;
}

// Exact BLEND_DEPTH order for one pixel of a long list, fragments read from
// HBM: rounds of a per-pixel window of the kSortWindow nearest (depth key,
// list index) keys above the last one blended, blended in that order.  The
// list arrives in (key, submit index) order, so ties on depth keep it.
template <int DT>
__device__ __forceinline__ void composite_exact(int n, const FragRec* list, uint64_t* kbAll,
                                                int t, int p, float& c0, float& c1, float& c2,
                                                float& al) {
  uint64_t* kb = kbAll + t;
  uint64_t lo = 0;
  int done = 0;
  while (done < n) {
    int m = 0;
    uint64_t last = 0;
    for (int ib = 0; ib < n; ib += 8) {
      float z[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) z[u] = (ib + u < n) ? __ldg(list[ib + u].depth + p) : 0.0f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = ib + u;
        if (i < n) {
          const uint64_t k = ((uint64_t)depth_bits(z[u]) << 32) | (uint32_t)i;
          if (done == 0 || k > lo) {
            if (m < kSortWindow) {
              if (m == 0 || k > last) {
                kb[m * kP] = k;
                last = k;
              } else {
                window_insert(kb, m, k);
              }
              ++m;
            } else if (k < last) {
              window_insert(kb, kSortWindow - 1, k);  // drops the largest
              last = kb[(kSortWindow - 1) * kP];
            }
          }
        }
      }
    }
    for (int r = 0; r < m; r += 4) {
      float4 c[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r + u < m) {
          const int i = (int)(uint32_t)kb[(r + u) * kP];
          c[u] = Px<DT>::global(list[i].rgba, p, list[i].scale);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (r + u < m) over(c[u], c0, c1, c2, al);
    }
    lo = last;
    done += m;
  }
}

// One pixel of one work item.
struct PixWork {
  const FrameArgs* A;
  int tile, chunk, p, P;
  bool active;
  uint32_t pix;   // row-major image index (frames hold at most 2^31 pixels)
  uint32_t sidx;  // tile-major state index (tile-major state of at most 2^32 pixels)
};

// `f`: the item's frame.
template <int FR>
__device__ __forceinline__ PixWork prepare(const FrameArgs* frames, const int* itemBase, int f,
                                           int item, int t) {
  PixWork w;
  const FrameArgs* A = frames + (FR == kOneFrame ? 0 : f);
  w.A = A;
  const int local = FR == kOneFrame ? item : item - itemBase[f];
  const int T = A->T;
  w.P = A->P;
  w.tile = local >> A->logChunks;
  w.chunk = local & (A->chunks - 1);
  // tile / tilesX without a division: (tile + 0.5) / tilesX is never within
  // float rounding of an integer for tile counts below 2^20
  const int ty = __float2int_rz(((float)w.tile + 0.5f) * A->invTilesX);
  const int tx = w.tile - ty * A->tilesX;
  w.p = w.chunk * w.P + t;
  w.sidx = (uint32_t)w.tile * (uint32_t)(T * T) + (uint32_t)w.p;
  const int x = tx * T + (w.p & (T - 1));
  const int y = ty * T + (w.p >> A->logT);
  w.active = (t < w.P) && (x < A->W) && (y < A->H);
  w.pix = (uint32_t)y * (uint32_t)A->W + (uint32_t)x;
  return w;
}

// Store, evict-first in L2 if `stream`.
template <class T>
__device__ __forceinline__ void put(T* p, T v, bool stream) {
  if (stream) __stcs(p, v); else *p = v;
}

// Background (generation 0), then the K4 epilogue of one pixel: colour,
// running sum (Kahan-compensated past the threshold), Welford M2, mean, RGBA8,
// and one variance partial per warp of 32 pixels.  S, M, CP are the pixel's
// previous sum, M2 and compensation.  Every lane of the warp calls it (the
// partial is a warp reduction); inactive lanes contribute zero.
template <int FR>
__device__ __forceinline__ void finish_pixel(const FrameArgs* A, const PixWork& w, int lane,
                                             int warp, float c0, float c1, float c2, float al,
                                             bool covered, float4 S, float4 M, float4 CP,
                                             const SrgbTables* tb, unsigned* err) {
  const unsigned flags = A->flags;
  const bool acc = (flags & DFB_FLAG_ACCUMULATE) != 0;
  float vsum = 0.0f;
  if (w.active) {
    if (A->mode != DFB_ZCOMPOSITE) {
      over(make_float4(A->bgR, A->bgG, A->bgB, A->bgA), c0, c1, c2, al);  // generation 0
    } else if (!covered) {
      c0 = A->bgR; c1 = A->bgG; c2 = A->bgB; al = A->bgA;
    }
    const float4 col = make_float4(c0, c1, c2, al);
    const bool pixOk = DFB_CHECK(w.pix < (size_t)A->W * A->H, err);
    const bool stateOk = DFB_CHECK(w.sidx < (size_t)A->nTiles * A->T * A->T, err);
    // images stream in frames that keep part of their state in L2, but not in
    // the first, which is often the only one and read back next (1920x1080
    // with its read-back: 62.7 us, 65.8 streamed)
    const bool stream = kKeeps<FR> && A->keepTiles != kKeepAll && A->frameN != 1;
    const bool streamState = kKeeps<FR> && w.tile >= A->keepTiles;
    if ((flags & DFB_FLAG_WRITE_COLOR) && pixOk) put(A->color + w.pix, col, stream);
    float4 out = col;
    if (acc) {
      float4 Sn, tot;
      if (A->kahan) {
        float4 cn;
#define DFB_KAHAN(ch)                 \
  {                                   \
    const float yk = col.ch - CP.ch;  \
    const float tk = S.ch + yk;       \
    cn.ch = (tk - S.ch) - yk;         \
    Sn.ch = tk;                       \
    tot.ch = tk - cn.ch;              \
  }
        DFB_KAHAN(x) DFB_KAHAN(y) DFB_KAHAN(z) DFB_KAHAN(w)
#undef DFB_KAHAN
        if (stateOk) put(A->comp + w.sidx, cn, streamState);
      } else {
        Sn = make_float4(S.x + col.x, S.y + col.y, S.z + col.z, S.w + col.w);
        tot = Sn;
      }
      const float iN = A->invN, iN1 = A->invNm1;
      const float4 mean = make_float4(tot.x * iN, tot.y * iN, tot.z * iN, tot.w * iN);
      if (A->frameN != 1) {
        // Welford: M2 += (x - mean_{n-1}) (x - mean_n), mean_{n-1} = S_{n-1}/(n-1)
        M.x = fmaf(col.x - S.x * iN1, col.x - mean.x, M.x);
        M.y = fmaf(col.y - S.y * iN1, col.y - mean.y, M.y);
        M.z = fmaf(col.z - S.z * iN1, col.z - mean.z, M.z);
        M.w = fmaf(col.w - S.w * iN1, col.w - mean.w, M.w);
      }
      if (stateOk) {
        put(A->accum + w.sidx, Sn, streamState);
        put(A->m2 + w.sidx, M, streamState);
      }
      vsum = (M.x + M.y + M.z) * iN1;
      out = mean;
    }
    if ((flags & DFB_FLAG_PACK_RGBA8) && pixOk)
      put(A->rgba8 + w.pix, pack_rgba8(pixel_op(out, A), tb), stream);
  }
  if (acc && warp * 32 < w.P) {
    // one partial per warp of 32 pixels, summed per tile by k_tile_variance
    float v = vsum;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const size_t slot = (size_t)w.tile * A->slots + ((w.chunk * w.P + warp * 32) >> 5);
    if (lane == 0 && DFB_CHECK(slot < (size_t)A->nTiles * A->slots, err)) A->varPartial[slot] = v;
  }
}

// A multi-fill item's fills, for one blend mode: the consumer group takes
// them from its slots in order (jg counts its fills) and carries the
// per-pixel blend across them; streamed state rows come with the last fill.
// BLEND_DEPTH blends speculatively in list order; `exact` turns false for a
// pixel whose finite depths are out of list order or that has a non-zero
// empty fragment.  Returns false when a wait ran out.
template <int DT, int MODE, int G>
__device__ __forceinline__ bool multi_fill(int total, const PixWork& w, int t, int lane,
                                           const LaunchCtl& ctl, unsigned char* ring,
                                           ItemMeta* metas, uint64_t* fullB, uint64_t* emptyB,
                                           volatile int* abort, uint32_t ringBytes, int group,
                                           int& jg, uint32_t stateRows, float& c0, float& c1,
                                           float& c2, float& al, bool& covered, bool& exact,
                                           float4& S0, float4& M, float4& CP) {
  constexpr int S = kSlots / G;
  const int fills = (total + kFill - 1) / kFill;
  const int P = w.P;
  float last = -INFINITY;
  uint32_t rest = 0u;
  bool bad = false;
  float zBest = INFINITY;
  const void* bestRgba = nullptr;
  float bestScale = 1.0f;
  for (int f = 0; f < fills; ++f) {
    const int s = group * S + jg % S;
    if (f > 0 && !wait_phase(&fullB[s], (uint32_t)(jg / S) & 1u, ctl, abort)) {
      if (lane == 0) give_up(ctl, abort);
      return false;
    }
    const ItemMeta* meta = metas + s;
    const unsigned char* base = ring + meta->start;
    const int nf = meta->n;
    const bool lastFill = f == fills - 1;
    const bool inRing = DFB_CHECK(
        nf <= kN && (uint64_t)meta->start + meta->bytes +
                            (uint64_t)(lastFill ? stateRows : 0u) * P * 16u <=
                        ringBytes,
        ctl.err);
    if (w.active && inRing) {
      const float* sD = reinterpret_cast<const float*>(base);
      constexpr bool hasD = MODE == DFB_BLEND_DEPTH || MODE == DFB_ZCOMPOSITE;
      const unsigned char* sC = base + (hasD ? (size_t)nf * P * 4 : 0);
      if (MODE == DFB_BLEND_ORDERED || MODE == DFB_AVERAGE) {
        if (P == kP)
          blend_list<DT, MODE, true>(nf, P, sC, meta, t, c0, c1, c2, al);
        else
          blend_list<DT, MODE, false>(nf, P, sC, meta, t, c0, c1, c2, al);
      } else if (MODE == DFB_ZCOMPOSITE) {
        const int i = nearest<false>(nf, P, sD, t, zBest);
        if (i >= 0) {
          bestRgba = meta->rgba[i];
          bestScale = meta->scale[i];
        }
      } else {
        if (P == kP)
          blend_in_order<DT, true>(nf, P, base, meta, t, c0, c1, c2, al, last, bad, rest);
        else
          blend_in_order<DT, false>(nf, P, base, meta, t, c0, c1, c2, al, last, bad, rest);
      }
    }
    if (lastFill && stateRows && inRing) {
      const float4* sState = reinterpret_cast<const float4*>(base + meta->bytes);
      S0 = sState[t];
      M = sState[P + t];
      if (stateRows == 3u) CP = sState[2 * P + t];
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&emptyB[s]);
    ++jg;
  }
  if (MODE == DFB_AVERAGE) {
    const float kk = (float)total;
    c0 = __fdiv_rn(c0, kk); c1 = __fdiv_rn(c1, kk); c2 = __fdiv_rn(c2, kk); al = __fdiv_rn(al, kk);
  } else if (MODE == DFB_ZCOMPOSITE) {
    covered = bestRgba != nullptr;
    if (covered && w.active) {
      const float4 v = Px<DT>::global(bestRgba, w.p, bestScale);
      c0 = v.x; c1 = v.y; c2 = v.z; al = v.w;
    }
  } else if (MODE == DFB_BLEND_DEPTH) {
    exact = !bad && rest == 0u;
  }
  return true;
}

// The pixel's state before this frame (the frame accumulates and is not the
// first); FR's frames may choose what stays in L2.
template <int FR>
__device__ __forceinline__ void read_state(const FrameArgs* A, const PixWork& w, float4& S,
                                           float4& M, float4& CP) {
  const bool comp = A->kahan && !A->kahanFirst;
  if (kKeeps<FR> && w.tile >= A->keepTiles) {
    S = __ldcs(A->accum + w.sidx);
    M = __ldcs(A->m2 + w.sidx);
    if (comp) CP = __ldcs(A->comp + w.sidx);
  } else {
    S = A->accum[w.sidx];
    M = A->m2[w.sidx];
    if (comp) CP = A->comp[w.sidx];
  }
}

// Consumer group: one pixel per thread.  Its items' fills come from its own
// slots, in order.
template <int DT, int G, int PER, int FR>
__device__ void consumer(const FrameArgs* __restrict__ frames, const int* __restrict__ itemBase,
                         int nFrames, int totalItems, const LaunchCtl& ctl, unsigned char* ring,
                         ItemMeta* metas, uint64_t* fullB, uint64_t* emptyB, volatile int* abort,
                         const SrgbTables* tb, uint32_t ringBytes) {
  constexpr int S = kSlots / G;
  const int group = threadIdx.x / kP;
  const int t = threadIdx.x - group * kP;  // pixel of the item, 0 .. kP-1
  const int lane = t & 31, warp = t >> 5;
  int jg = 0;     // this group's fills taken
  int frame = 0;  // the item's frame
  const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
  // The pixel's accumulation state comes with the item's last fill, or, in
  // frames that do not stream it, is loaded by the consumer itself
  // (tile-major: each warp reads 512 contiguous bytes per buffer) at the
  // item's start, before the wait for its fragments.  For the narrow
  // storage formats in single-frame launches of 2 CTAs per SM with one
  // group, the loads are issued one item ahead -- while the group waits
  // for, blends and finishes the item before -- so that their latency is
  // hidden (FP16 at 5.5 fragments per tile: 0.1029 against 0.1058 ms).
  // Elsewhere that costs more than it hides: FP32 gains nothing, the
  // multi-frame launches pay a second frame search per item (batched graph
  // 1.99 against 1.74 ms), 3 CTAs per SM lose registers, and several groups
  // per CTA would spill.
  constexpr bool ahead = G == 1 && PER == 2 && FR == kOneFrame && DT != DFB_F32;
  auto load_state = [&](int it, float4& s0, float4& m2, float4& cp) {
    s0 = m2 = cp = zero4;
    if (it >= totalItems) return;
    const PixWork v = prepare<FR>(frames, itemBase, 0, it, t);  // single-frame launches only
    const FrameArgs* B = v.A;
    if (v.active && (B->flags & DFB_FLAG_ACCUMULATE) && B->frameN != 1 && !B->stateInRing &&
        DFB_CHECK(v.sidx < (size_t)B->nTiles * B->T * B->T, ctl.err))
      read_state<FR>(B, v, s0, m2, cp);
  };
  float4 nS0, nM, nCP;  // the next item's state (loads one item ahead)
  if constexpr (ahead) load_state(blockIdx.x, nS0, nM, nCP);
  for (int k = group; ; k += G) {
    const int item = blockIdx.x + k * (int)gridDim.x;
    if (item >= totalItems) break;
    frame = next_frame<FR>(itemBase, frame, item);
    const PixWork w = prepare<FR>(frames, itemBase, frame, item, t);
    const FrameArgs* A = w.A;
    const bool accRead = w.active && (A->flags & DFB_FLAG_ACCUMULATE) && A->frameN != 1 &&
                         DFB_CHECK(w.sidx < (size_t)A->nTiles * A->T * A->T, ctl.err);
    const uint32_t stateRows =
        accRead && A->stateInRing ? ((A->kahan && !A->kahanFirst) ? 3u : 2u) : 0u;
    float4 S0, M, CP;
    if constexpr (ahead) {
      S0 = nS0;
      M = nM;
      CP = nCP;
      load_state(item + (int)gridDim.x, nS0, nM, nCP);
    } else {
      S0 = M = CP = zero4;
      if (accRead && !A->stateInRing) read_state<FR>(A, w, S0, M, CP);
    }
    int s = group * S + jg % S;
    if (!wait_phase(&fullB[s], (uint32_t)(jg / S) & 1u, ctl, abort)) {
      if (lane == 0) give_up(ctl, abort);
      break;
    }
    const ItemMeta* meta = metas + s;
    const int total = meta->total;
    const int P = w.P;
    float c0 = 0.f, c1 = 0.f, c2 = 0.f, al = 0.f;
    bool covered = true;
    if (total <= kN) {
      const unsigned char* base = ring + meta->start;
      // checked build: the item's fragments and state rows lie inside the ring
      const bool inRing = DFB_CHECK(
          meta->n <= kN && (uint64_t)meta->start + meta->bytes + (uint64_t)stateRows * P * 16u <=
                               ringBytes,
          ctl.err);
      if (w.active && inRing)
        covered = P == kP ? composite_staged<DT, true>(item_mode(A->mode, total), total, P,
                                                       base, meta, t, w.p, c0, c1, c2, al)
                          : composite_staged<DT, false>(item_mode(A->mode, total), total, P,
                                                        base, meta, t, w.p, c0, c1, c2, al);
      // streamed state: from the ring into registers; then the ring space
      // goes back to the producer before the epilogue's math and stores
      if (stateRows && inRing) {
        const float4* sState = reinterpret_cast<const float4*>(base + meta->bytes);
        S0 = sState[t];
        M = sState[P + t];
        if (stateRows == 3u) CP = sState[2 * P + t];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&emptyB[s]);  // ring space free for the producer
      ++jg;
    } else {
      // multi-fill item: kFill fragments per fill
      bool ok, exact = true;
      switch (A->mode) {
        case DFB_BLEND_DEPTH:
          ok = multi_fill<DT, DFB_BLEND_DEPTH, G>(total, w, t, lane, ctl, ring, metas, fullB,
                                                  emptyB, abort, ringBytes, group, jg, stateRows,
                                                  c0, c1, c2, al, covered, exact, S0, M, CP);
          break;
        case DFB_BLEND_ORDERED:
          ok = multi_fill<DT, DFB_BLEND_ORDERED, G>(total, w, t, lane, ctl, ring, metas, fullB,
                                                    emptyB, abort, ringBytes, group, jg, stateRows,
                                                    c0, c1, c2, al, covered, exact, S0, M, CP);
          break;
        case DFB_ZCOMPOSITE:
          ok = multi_fill<DT, DFB_ZCOMPOSITE, G>(total, w, t, lane, ctl, ring, metas, fullB,
                                                 emptyB, abort, ringBytes, group, jg, stateRows,
                                                 c0, c1, c2, al, covered, exact, S0, M, CP);
          break;
        default:
          ok = multi_fill<DT, DFB_AVERAGE, G>(total, w, t, lane, ctl, ring, metas, fullB, emptyB,
                                              abort, ringBytes, group, jg, stateRows, c0, c1,
                                              c2, al, covered, exact, S0, M, CP);
          break;
      }
      if (!ok) break;
      if (__any_sync(0xffffffffu, w.active && !exact)) {
        // out-of-order depths (or a non-zero empty fragment) in this warp's
        // 32 pixels: the exact re-do kernel composites them after this launch
        if (lane == 0) {
          const int slot = atomicAdd(ctl.redo, 1);
          ctl.redo[1 + slot] = item * (kP / 32) + warp;
        }
        continue;
      }
    }
    finish_pixel<FR>(A, w, lane, warp, c0, c1, c2, al, covered, S0, M, CP, tb, ctl.err);
  }
}

// FR = kOneFrame: a single-frame launch, whose arguments come as the kernel
// parameter `prm`; kParamTable: the frame table (and work-item prefix) of a
// launch of at most kParamFrames frames comes as `prm`; both are read from
// the parameter space.  kGlobalTable: `frames` and `itemBase` are the
// launch's tables in global memory.
template <int DT, int G, int PER, int FR>
__global__ void __launch_bounds__(Shape<G>::threads, PER)
    k_composite(const FrameArgs* __restrict__ frames, const int* __restrict__ itemBase,
                int nFrames, int totalItems, uint32_t ringBytes, LaunchCtl ctl,
                const __grid_constant__ typename FrameParams<FR>::type prm) {
  if constexpr (FR == kOneFrame) frames = &prm;
  if constexpr (FR == kParamTable) {
    frames = prm.f;
    itemBase = prm.itemBase;
  }
  extern __shared__ __align__(128) unsigned char smem[];
  SrgbTables* tb = reinterpret_cast<SrgbTables*>(smem);
  uint64_t* fullB = reinterpret_cast<uint64_t*>(smem + kOffBars);
  uint64_t* emptyB = fullB + kSlots;
  volatile int* abort = reinterpret_cast<volatile int*>(smem + kOffFlags);
  ItemMeta* metas = reinterpret_cast<ItemMeta*>(smem + kOffMetas);
  TileBlock* queue = reinterpret_cast<TileBlock*>(smem + kOffQueue);
  uint64_t* queueB = emptyB + kSlots;
  unsigned char* ring = smem + kHeader;
  load_srgb(tb, Shape<G>::threads);
  if (threadIdx.x == 0) {
    for (int q = 0; q < kSlots; ++q) {
      mbar_init(&fullB[q], 1);
      mbar_init(&emptyB[q], kCW);
    }
    for (int q = 0; q < 2; ++q) mbar_init(&queueB[q], 1);
    *abort = 0;
    fence_barrier_init();
  }
  // The set-up above reads nothing that earlier kernels write; with a
  // programmatic launch it overlaps the end of the kernel before.
  grid_dependency_wait();
  allow_dependents();
  __syncthreads();
  if (threadIdx.x >= G * kP)
    producer<DT, G, FR>(frames, itemBase, nFrames, totalItems, ctl, ring, ringBytes, metas, queue,
                        fullB, emptyB, queueB, abort);
  else
    consumer<DT, G, PER, FR>(frames, itemBase, nFrames, totalItems, ctl, ring, metas, fullB,
                             emptyB, abort, tb, ringBytes);
}

// A warp's scratch of the exact re-do: the fragments of one unit's list.
struct RedoWarp {
  const void* rgba[kRedoRank];
  const float* depth[kRedoRank];
  float scale[kRedoRank];
  float z[kRedoRank][32];               // canonical depths, a column per pixel
  unsigned char order[kRedoRank][32];   // fragment of each place in the pixel's order
};

// Exact BLEND_DEPTH order for one pixel of a list of at most kRedoRank
// fragments: all depths are read once, several in flight, a fragment's place
// is the number of fragments before it by (depth, list index), and the RGBA
// are read in that order, several in flight.  Called by the active lanes of a
// warp; `w` holds the list's pointers already.
template <int DT>
__device__ __forceinline__ void composite_ranked(int n, RedoWarp* w, int lane, int p, float& c0,
                                                 float& c1, float& c2, float& al) {
  for (int i0 = 0; i0 < n; i0 += 8) {
    float z[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i0 + u < n) z[u] = __ldg(w->depth[i0 + u] + p);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i0 + u < n) w->z[i0 + u][lane] = covers(z[u]) ? z[u] : INFINITY;
  }
  for (int i0 = 0; i0 < n; i0 += 4) {
    float z[4];
    int rank[4] = {0, 0, 0, 0};
#pragma unroll
    for (int u = 0; u < 4; ++u) z[u] = i0 + u < n ? w->z[i0 + u][lane] : INFINITY;
#pragma unroll 4
    for (int j = 0; j < i0; ++j) {
      const float v = w->z[j][lane];
#pragma unroll
      for (int u = 0; u < 4; ++u) rank[u] += v <= z[u] ? 1 : 0;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + j < n && j != u) rank[u] += (j < u ? z[j] <= z[u] : z[j] < z[u]) ? 1 : 0;
#pragma unroll 4
    for (int j = i0 + 4; j < n; ++j) {
      const float v = w->z[j][lane];
#pragma unroll
      for (int u = 0; u < 4; ++u) rank[u] += v < z[u] ? 1 : 0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u < n) w->order[rank[u]][lane] = (unsigned char)(i0 + u);
  }
  for (int r0 = 0; r0 < n; r0 += 4) {
    float4 f[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (r0 + u < n) {
        const int i = w->order[r0 + u][lane];
        f[u] = Px<DT>::global(w->rgba[i], p, w->scale[i]);
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (r0 + u < n) over(f[u], c0, c1, c2, al);
  }
}

// Exact re-do of the 32-pixel units (work item, warp) that the persistent
// kernel left: multi-fill BLEND_DEPTH items whose depths were out of list
// order at some pixel, or that had a non-zero empty fragment.  Each warp of a
// CTA takes one unit at a time; each pixel reads its fragments from memory
// (mostly still in L2) and blends them in exact (depth, key, submit index)
// order, then goes through the same epilogue.  Where the keys follow the
// depths (bricks) there are no units and the kernel returns at once; where
// producers overlap, most units of a long list are here.
//
// Two kernels, each for its own units; a launch runs those it has lists for:
//   * RANKED: lists of up to kRedoRank fragments, by rank.  Bound by the
//     latency of its dependent reads, so warps matter more than reads in
//     flight per warp: kRedoPer CTAs per SM (their scratch fills its shared
//     memory), 8 depths and 4 RGBA per lane at a time.  A 1024x1024 FP32 frame
//     with 3,500 units of 17 to 24 fragments takes 88 us with its read-back;
//     6 us more with 2 CTAs per SM and twice the reads in flight or not, or
//     when the warps of a CTA wait for one another; 41 against 31 us of this
//     kernel by windowed rounds.  Launched programmatically, so that a launch
//     that finds no units costs no more than its own start: 16 passes of FP8
//     4096x1024 1.435 -> 1.396 ms.
//   * longer lists, by the windowed rounds of composite_exact.  As a call
//     within the other kernel, whose warps then waited for one another, they
//     were slower: a 512x512 FP32 frame out of order everywhere, 49 fragments
//     per tile 704 us, 471 so; 150 per tile 4181 and 3173.  Launched plainly:
//     with a programmatic launch, whose CTAs are placed while the composite
//     still holds most SMs, the same frames take 640 and 3850 us.
template <int DT, bool RANKED>
__global__ void __launch_bounds__(kP, RANKED ? kRedoPer : kWindowPer) k_composite_redo(
    const FrameArgs* __restrict__ frames, const int* __restrict__ itemBase, int nFrames,
    LaunchCtl ctl) {
  extern __shared__ __align__(128) unsigned char lsmem[];
  SrgbTables* tb = reinterpret_cast<SrgbTables*>(lsmem);
  grid_dependency_wait();  // the composite's list of units, and its writes
  allow_dependents();
  const int count = *(volatile int*)ctl.redo;
  if ((int)blockIdx.x * kCW >= count) return;
  load_srgb(tb, kP);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int u = blockIdx.x * kCW + warp; u < count; u += gridDim.x * kCW) {
    const int entry = ctl.redo[1 + u];
    const int item = entry / kCW, iw = entry % kCW;
    const int f = find_frame(itemBase, nFrames, item);
    const int local = item - __ldg(itemBase + f);
    const FrameArgs* A = frames + f;
    if (!DFB_CHECK(f >= 0 && f < nFrames && (local >> A->logChunks) < A->nTiles, ctl.err))
      continue;
    const TileBlock* blk = A->blocks + A->tileBase + (local >> A->logChunks);
    const int n = blk->n;
    if ((n <= kRedoRank) != RANKED) continue;
    const FragRec* list = A->srecs + blk->off;
    const PixWork w = prepare<kGlobalTable>(frames, itemBase, f, item, iw * 32 + lane);
    float c0 = 0.f, c1 = 0.f, c2 = 0.f, al = 0.f;
    if constexpr (RANKED) {
      RedoWarp* rw = reinterpret_cast<RedoWarp*>(lsmem + sizeof(SrgbTables)) + warp;
      for (int i = lane; i < n; i += 32) {
        rw->rgba[i] = list[i].rgba;
        rw->depth[i] = list[i].depth;
        rw->scale[i] = list[i].scale;
      }
      __syncwarp();
      if (w.active) composite_ranked<DT>(n, rw, lane, w.p, c0, c1, c2, al);
      __syncwarp();
    } else {
      uint64_t* window = reinterpret_cast<uint64_t*>(lsmem + sizeof(SrgbTables));
      if (w.active) composite_exact<DT>(n, list, window, threadIdx.x, w.p, c0, c1, c2, al);
    }
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 S = zero4, M = zero4, CP = zero4;
    if (w.active && (A->flags & DFB_FLAG_ACCUMULATE) && A->frameN != 1)
      read_state<kGlobalTable>(A, w, S, M, CP);
    finish_pixel<kGlobalTable>(A, w, lane, iw, c0, c1, c2, al, true, S, M, CP, tb, ctl.err);
  }
}

// Per-tile variance of one frame's tile: a warp sums the tile's per-warp
// partials in slot order.
__device__ __forceinline__ void tile_variance(const FrameArgs* A, int tile, int lane) {
  const int slots = A->slots;
  float sum = 0.0f;
  for (int q = lane; q < slots; q += 32) sum += A->varPartial[(size_t)tile * slots + q];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) {
    const int T = A->T;
    const int tx = tile % A->tilesX, ty = tile / A->tilesX;
    const int w = min(T, A->W - tx * T), h = min(T, A->H - ty * T);
    A->tileVar[tile] = sum / (3.0f * (float)(w * h));
  }
}

// One warp per global tile of a launch over several frames.
__global__ void k_tile_variance(const FrameArgs* __restrict__ frames, int nFrames,
                                int totalTiles) {
  grid_dependency_wait();  // the composite's partials
  allow_dependents();
  const int gt = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
  if (gt >= totalTiles) return;
  int lo = 0, hi = nFrames - 1;  // frame with the largest tileBase <= gt
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (frames[mid].tileBase <= gt) lo = mid; else hi = mid - 1;
  }
  const FrameArgs* A = frames + lo;
  if (A->flags & DFB_FLAG_ACCUMULATE) tile_variance(A, gt - A->tileBase, threadIdx.x & 31);
}

// The same for a single frame, whose arguments come with the launch: between
// two composites this kernel is a chain of dependent loads, and the two from
// the frame table are gone (16 passes of FP8 4096x1024 1.388 -> 1.382 ms).
__global__ void k_tile_variance_one(const __grid_constant__ FrameArgs frame) {
  grid_dependency_wait();
  allow_dependents();
  const int tile = (int)((blockIdx.x * (unsigned)blockDim.x + threadIdx.x) >> 5);
  if (tile < frame.nTiles) tile_variance(&frame, tile, threadIdx.x & 31);
}

template <int DT, int G, int PER>
cudaError_t launch_shape(const FrameArgs* frames, const int* itemBase, int nFrames,
                         int totalItems, int ringKB, const LaunchCtl& ctl,
                         const FrameArgs* hostFrames, const int* hostItemBase, cudaStream_t s) {
  auto kTable = k_composite<DT, G, PER, kGlobalTable>;
  auto kOne = k_composite<DT, G, PER, kOneFrame>;
  auto kParam = k_composite<DT, G, PER, kParamTable>;
  constexpr int per = PER;  // CTAs per SM
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  static int sms[64] = {0};
  static int smemMax[64] = {0};
  if (!sms[dev]) {
    int optin = 0, perSm = 0;
    e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
      e = cudaDeviceGetAttribute(&perSm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kTable, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kOne, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kParam, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e != cudaSuccess) {
      sms[dev] = 0;
      return e;
    }
    // per CTA: what `per` CTAs can share, less the 1 KB of shared memory CUDA
    // reserves for each CTA
    const int share = perSm / per - 1024;
    smemMax[dev] = share < optin ? share : optin;
  }
  uint32_t ring = (uint32_t)ringKB * 1024u;
  const uint32_t cap = (uint32_t)(smemMax[dev] - kHeader) & ~127u;
  if (ring > cap) ring = cap;
  if (ring < Bytes<DT>::maxItem) return cudaErrorInvalidConfiguration;
  int grid = sms[dev] * per;
  if (grid > totalItems) grid = totalItems;
  if (grid < 1) return cudaSuccess;
  const size_t smem = kHeader + ring;
  if (hostFrames && nFrames == 1)
    return launch_programmatic(kOne, grid, Shape<G>::threads, smem, s, frames, itemBase, nFrames,
                               totalItems, ring, ctl, hostFrames[0]);
  if (hostFrames && hostItemBase && nFrames <= kParamFrames) {
    FrameTable tab;
    memcpy(tab.itemBase, hostItemBase, sizeof(int) * (nFrames + 1));
    memcpy(tab.f, hostFrames, sizeof(FrameArgs) * nFrames);
    return launch_programmatic(kParam, grid, Shape<G>::threads, smem, s, frames, itemBase,
                               nFrames, totalItems, ring, ctl, tab);
  }
  return launch_programmatic(kTable, grid, Shape<G>::threads, smem, s, frames, itemBase, nFrames,
                             totalItems, ring, ctl, 0);
}

constexpr int kRankedSmem = (int)(sizeof(SrgbTables) + sizeof(RedoWarp) * kCW);
constexpr int kWindowSmem = (int)(sizeof(SrgbTables) + kWindowBytes);

// One-time set-up of a format's re-do kernels on the current device.
template <int DT>
cudaError_t redo_setup() {
  const cudaError_t e = cudaFuncSetAttribute(
      k_composite_redo<DT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRankedSmem);
  return e != cudaSuccess
             ? e
             : cudaFuncSetAttribute(k_composite_redo<DT, false>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, kWindowSmem);
}

// The re-do of a launch's long lists: at most one unit per warp of their
// items; the count is on the device.
template <int DT>
cudaError_t launch_redo(const FrameArgs* frames, const int* itemBase, int nFrames,
                        const LaunchCtl& ctl, const LongList& lng, int sms, cudaStream_t s) {
  const int items = lng.ranked + lng.windowed;
  auto grid = [&](int per) { return items < per * sms ? items : per * sms; };
  cudaError_t e = cudaSuccess;
  if (lng.ranked > 0)
    e = launch_programmatic(k_composite_redo<DT, true>, grid(kRedoPer), kP, kRankedSmem, s, frames,
                            itemBase, nFrames, ctl);
  if (e == cudaSuccess && lng.windowed > 0) {
    k_composite_redo<DT, false><<<grid(kWindowPer), kP, kWindowSmem, s>>>(frames, itemBase,
                                                                         nFrames, ctl);
    e = cudaGetLastError();
  }
  return e;
}

template <int DT>
cudaError_t launch_dt(const FrameArgs* frames, const int* itemBase, int nFrames, int totalItems,
                      const TuneParams& tune, const LaunchCtl& ctl, const FrameArgs* hostFrames,
                      const int* hostItemBase, cudaStream_t s) {
  const int per = tune.ctasPerSm, g = tune.groups;
#define DFB_SHAPE(G_, PER_)                                                                   \
  if (g == G_ && per == PER_)                                                                 \
    return launch_shape<DT, G_, PER_>(frames, itemBase, nFrames, totalItems, tune.ringKB, ctl,  \
                                      hostFrames, hostItemBase, s);
  DFB_SHAPE(1, 2)
  DFB_SHAPE(2, 2)
  DFB_SHAPE(1, 3)
  DFB_SHAPE(2, 1)
  DFB_SHAPE(3, 1)
#undef DFB_SHAPE
  return cudaErrorInvalidConfiguration;
}

}  // namespace

// Measured (composite launch): FP32 takes 2 CTAs per SM with one consumer
// group each and the largest ring they share; its largest fill does not fit
// the rings of 3.  The narrower formats' does, and 3 CTAs per SM are faster:
// FP8 4096x1024, 3.4 fragments per tile, accumulating, 82 against 88 us; 16
// mixed FP16 frames of 2 to 25 per tile in one launch 634 against 708 us.  The
// exception are single FP16 and BF16 frames from 5 fragments per tile:
// 2048x2048, 5.5 per tile, accumulating 102.0 against 107.3 us (4.4 per tile:
// 102.8 against 94.5), not accumulating 6 per tile 90.9 against 97.7; FP8
// would be faster with 3 there too (98 against 91 us).
// A ring of 70 KB beats the largest (103.6 us) as long as it holds two items
// and more: further reads in flight than the DRAM queues need only spread the
// accesses to a tile in time.  At 8 per tile in every tile it takes 104 against
// 112 us; at 12, where it holds one item, 167 against 132; in frames of bricks,
// whose tiles differ, 117 and 117 at 7.7 per tile, 135 and 132 at 9.7, 154 and
// 147 at 11.9.  So it is taken up to 8.  One CTA per SM is slower everywhere:
// its single producer warp sets the pace.
TuneParams default_tune(int dtype, double fragmentsPerTile, bool oneFrame) {
  if (dtype == DFB_F32) return TuneParams{110, 2, 1};
  if (oneFrame && fragmentsPerTile >= 5.0)
    return TuneParams{fragmentsPerTile <= 8.0 ? 70 : 110, 2, 1};
  return TuneParams{72, 3, 1};
}

cudaError_t launch_composite(const FrameArgs* frames, const int* itemBase, int nFrames,
                             int totalItems, int totalTiles, bool accumulate, int dtype,
                             const TuneParams& tune, const LaunchCtl& ctl, const LongList& lng,
                             const FrameArgs* hostFrames, const int* hostItemBase,
                             cudaEvent_t afterMain, cudaStream_t s) {
  cudaError_t e;
  switch (dtype) {
    case DFB_F32:
      e = launch_dt<DFB_F32>(frames, itemBase, nFrames, totalItems, tune, ctl, hostFrames,
                                 hostItemBase, s);
      break;
    case DFB_F16:
      e = launch_dt<DFB_F16>(frames, itemBase, nFrames, totalItems, tune, ctl, hostFrames,
                                 hostItemBase, s);
      break;
    case DFB_BF16:
      e = launch_dt<DFB_BF16>(frames, itemBase, nFrames, totalItems, tune, ctl, hostFrames,
                                 hostItemBase, s);
      break;
    default:
      e = launch_dt<DFB_FP8E4M3>(frames, itemBase, nFrames, totalItems, tune, ctl, hostFrames,
                                 hostItemBase, s);
      break;
  }
  if (e == cudaSuccess && afterMain) e = cudaEventRecord(afterMain, s);
  // One-time set-up of the re-do kernel per device, done on any launch (so
  // that it never first happens inside a stream capture).
  static int sms[64] = {0};
  int dev = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess && (dev < 0 || dev >= 64)) e = cudaErrorInvalidDevice;
  if (e == cudaSuccess && !sms[dev]) {
    int count = 0;
    e = cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = redo_setup<DFB_F32>();
    if (e == cudaSuccess) e = redo_setup<DFB_F16>();
    if (e == cudaSuccess) e = redo_setup<DFB_BF16>();
    if (e == cudaSuccess) e = redo_setup<DFB_FP8E4M3>();
    if (e == cudaSuccess) sms[dev] = count;
  }
  if (e == cudaSuccess && lng.kernels()) {
    auto redo = launch_redo<DFB_FP8E4M3>;
    if (dtype == DFB_F32) redo = launch_redo<DFB_F32>;
    if (dtype == DFB_F16) redo = launch_redo<DFB_F16>;
    if (dtype == DFB_BF16) redo = launch_redo<DFB_BF16>;
    e = redo(frames, itemBase, nFrames, ctl, lng, sms[dev], s);
  }
  if (e != cudaSuccess || !accumulate || totalTiles < 1) return e;
  const int grid = (totalTiles * 32 + 255) / 256;
  if (hostFrames && nFrames == 1)
    return launch_programmatic(k_tile_variance_one, grid, 256, 0, s, hostFrames[0]);
  return launch_programmatic(k_tile_variance, grid, 256, 0, s, frames, nFrames, totalTiles);
}

}  // namespace dfb
