// Shared definitions for the libnsml device code (sm_100a).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include "nsml.h"
#include "nsml_plan.h"

namespace nsml {

// Radix digits of the 31-bit magnitude key, most significant first:
// bits 30..19 (8 exponent + 4 mantissa bits), bits 18..7, bits 6..0.
__host__ __device__ constexpr int digit_bits(int level) { return level == 2 ? 7 : 12; }
__host__ __device__ constexpr int digit_shift(int level) { return level == 0 ? 19 : (level == 1 ? 7 : 0); }
constexpr int kMaxBins = 4096;

constexpr int kCta = 256;          // threads per block in every streaming kernel
constexpr uint32_t kInfKey = 0x7F800000u;

// Polls before a wait at a grid barrier gives up (each poll sleeps a little,
// so this is on the order of a second).
constexpr int kMaxPolls = 1 << 22;

// Control block at the start of a compress workspace.  Cleared (together with
// the histograms that follow it) at the start of every call.
struct Ctl {
  int status;                 // first device-detected error (NSML_ERR_*), 0 = ok
  unsigned int lo, hi;        // sampled bounds of the threshold key: probably lo <= T < hi
  unsigned int barrier;       // arrivals at the grid barriers of a cooperative kernel
  unsigned int grain;         // the sampled keys (nearly all of them) are multiples of 1 << grain: 16, 13 or 0
  unsigned int ticket;        // chunks of the list handed out
  unsigned int fallback;      // a bin that was taken for a single key holds others
  unsigned int done;          // chunks of the list that are finished, where that has to be known
  unsigned long long below_listed;     // mask build: weights below the bracket << 32 | weights listed inside it
  unsigned int drawn[9], finished[9];  // general select, mask build: units of work of each phase
  unsigned long long listed_above;  // grid select: candidates << 32 | those above the window
  unsigned int sampled, members;    // grid select: sampler blocks done; keys of the threshold's bin
  unsigned int zeros[4];            // grid select: zeros among the keys that the histogram of a round counted
};
static_assert(sizeof(Ctl) <= 256, "control block must fit its 256-byte slot");

// The window of keys the sample leaves open, cut into at most kMaxBins bins of 1 << shift keys.
struct Window {
  unsigned int lo, hi, shift;  // keys lo .. hi-1; bin (key - lo) >> shift
  unsigned int grain;          // the keys are (taken to be) multiples of 1 << grain
  bool few;                    // there are at most kFewBins bins

  __device__ __forceinline__ bool single() const { return shift <= grain; }  // a bin holds one key ...
  __device__ __forceinline__ unsigned int key_of(unsigned int bin) const {   // ... this one
    return (lo + (bin << shift) + ((1u << grain) - 1u)) & ~((1u << grain) - 1u);
  }
};
constexpr unsigned int kFewBins = 64;
// TYPE: element type of the keys.  The low 16 bits of a bfloat16 key are zero, so a bin need not be narrower than that
// and holds one key then; the same goes for float32 buckets widened from bfloat16 or binary16 (13 bits), which the
// sample tells and the list stage verifies.
template <int TYPE>
__host__ __device__ constexpr unsigned int min_bin_shift() { return TYPE == NSML_F32 ? 0 : 16; }
template <int TYPE>
__device__ __forceinline__ Window make_window(const Ctl* ctl) {
  Window w;
  const unsigned int hi = ctl->hi;
  w.grain = TYPE == NSML_BF16 ? 16u : ctl->grain;
  // 0: the sample holds too few non-zero keys; everything is listed, zeros too.  At most infinity: a bucket with many
  // NaN has a NaN's key here, and the bucket pass compares floats with it, so that it would list every key and count
  // those below `lo` in bins that do not exist.
  w.lo = min(ctl->lo, kInfKey);
  w.hi = hi > w.lo ? hi : 0x80000000u;
  const unsigned int span = (w.hi - w.lo - 1) / kMaxBins;
  w.shift = max(w.grain, span == 0 ? 0u : 32u - __clz(span));
  w.few = (w.hi - w.lo - 1) >> w.shift < kFewBins;
  return w;
}

constexpr int kTileBytes = 16384;         // bucket bytes per tile of the candidate list: what a block of the bucket pass takes
constexpr int kMaxGroups = 8192;          // the bucket pass keeps a candidate count per group of tiles (of one tile, up to 32M
                                          // float32 or 64M bfloat16 elements)
constexpr int kChunk = 2048;              // candidates a block of the list stage takes at a time (long lists: twice that)

// The keys inside the window are also kept by bin, up to this many per bin: four times what is to be expected where the
// window is widest (kept fraction a quarter: 2 per cent of the bucket over at least 2048 bins).
inline unsigned int bin_room_of(int64_t n) {
  unsigned int room = 16;
  while (room < 2048 && (int64_t)room * 25000 < n) room *= 2;
  return room;
}

// elements per tile; TYPE: element type of the stream the tiles cut (a tile of a bucket with a residual holds
// float32 sums)
template <int TYPE>
__host__ __device__ constexpr int tile_elems() { return kTileBytes / (TYPE == NSML_F32 ? 4 : 2); }
// tiles per group, as a shift
inline unsigned int group_shift_of(unsigned long long tiles) {
  unsigned int s = 0;
  while (((tiles + (1ull << s) - 1) >> s) > (unsigned long long)kMaxGroups) ++s;
  return s;
}

struct CompressLayout {  // byte offsets inside a compress workspace
  size_t hist;          // u32[4][kMaxBins]: digit histograms; the last one counts the candidates inside the sampled window
  size_t group_count;   // u32[kMaxGroups]: candidates per group of tiles
  size_t zero_bytes;    // everything before this offset is cleared per call
  size_t bins;          // uint2[kMaxBins][bin_room_of(n)]: (key, index) of the candidates inside the window, by bin
  size_t chunk_sum;     // u64[2][chunks]: survivors of a chunk, and up to it; cleared by the bucket pass
  size_t block_fill;    // u32[chunks]: values delivered to a payload block of 1024; cleared by the bucket pass
  size_t tile_count;    // u32[tiles]: candidates per tile
  size_t cand_off;      // u16[n]: a candidate's offset inside its tile; tile t's candidates start at t * tile_elems
  size_t cand_val;      // u32[n]: float32 bit patterns (bfloat16 bucket: offset << 16 | bfloat16 bits, and no cand_off)
  size_t raw_val;       // f32[n]: survivor values before int8 quantisation
  size_t total;
};

inline CompressLayout compress_layout(int64_t n) {
  CompressLayout L;
  const size_t npad = align_up((size_t)n, tile_elems<NSML_BF16>());
  L.hist = 256;
  L.group_count = L.hist + 4 * kMaxBins * sizeof(unsigned int);
  L.zero_bytes = L.group_count + kMaxGroups * sizeof(unsigned int);
  L.bins = L.zero_bytes;
  L.chunk_sum = L.bins + (size_t)kMaxBins * bin_room_of(n) * 8;
  const size_t chunks = npad / kChunk;
  L.block_fill = L.chunk_sum + align_up(2 * chunks * 8, 256);
  L.tile_count = L.block_fill + align_up(chunks * 4, 256);
  L.cand_off = L.tile_count + align_up(npad / tile_elems<NSML_F32>() * 4, 256);
  L.cand_val = L.cand_off + npad * 2;
  L.raw_val = L.cand_val + npad * 4;
  L.total = L.raw_val + npad * 4;
  return L;
}

struct PayloadLayout {
  int64_t k;
  size_t idx_off, val_off, scale_off, nblocks, total;
};

inline PayloadLayout payload_layout(int64_t k, int bits) {
  PayloadLayout P;
  P.k = k;
  P.idx_off = sizeof(nsml_payload_header);
  P.val_off = P.idx_off + align_up((size_t)k * 4, 16);
  if (bits == NSML_BITS_INT8) {
    P.nblocks = (size_t)((k + NSML_QBLOCK - 1) / NSML_QBLOCK);
    P.scale_off = P.val_off + align_up((size_t)k, 16);
    P.total = P.scale_off + align_up(P.nblocks * 4, 16);
  } else {  // fp16: 2 bytes per value; float32 as is: 4
    P.nblocks = 0;
    P.scale_off = 0;
    P.total = P.val_off + align_up((size_t)k * (bits == NSML_BITS_FP32 ? 4 : 2), 16);
  }
  return P;
}

__device__ __forceinline__ void set_status(int* status, int code) { atomicCAS(status, 0, code); }

// ---- programmatic dependent launch: a kernel launched with the attribute may start while its predecessor in the
// stream still runs; pdl_wait returns when the predecessor has completed and its writes are visible.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---- bulk copy shared -> global by one thread (16-byte aligned addresses and size) ----
// Writers of the shared memory call fence_async_shared, then the block synchronises, then one thread stores.
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void bulk_store(void* gdst, const void* smem_src, unsigned int bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst),
               "r"((uint32_t)__cvta_generic_to_shared(smem_src)), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// ------------------------------------------------------------------------
// Element sources.  load_vals4 returns the float32 bit patterns of elements
// i0..i0+3 (i0 a multiple of 4) and how many of them exist (0..4); missing
// ones read as 0.  Pruned elements (mask bit set) read as +0.0.
// ------------------------------------------------------------------------
template <int DTYPE>
struct BucketSrc {
  const void* grad;
  const uint32_t* mask;  // may be null

  __device__ __forceinline__ int load_vals4(unsigned long long i0, unsigned long long count, uint32_t (&bits)[4]) const {
    int cnt;
    if (i0 + 4 <= count) {
      if (DTYPE == NSML_F32) {
        const uint4 v = __ldcs(reinterpret_cast<const uint4*>(static_cast<const uint32_t*>(grad) + i0));
        bits[0] = v.x; bits[1] = v.y; bits[2] = v.z; bits[3] = v.w;
      } else {
        const uint2 v = __ldcs(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(grad) + i0));
        bits[0] = v.x << 16; bits[1] = v.x & 0xFFFF0000u;
        bits[2] = v.y << 16; bits[3] = v.y & 0xFFFF0000u;
      }
      cnt = 4;
    } else {
      cnt = (i0 < count) ? (int)(count - i0) : 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        bits[e] = 0;
        if (e < cnt) {
          if (DTYPE == NSML_F32) bits[e] = static_cast<const uint32_t*>(grad)[i0 + e];
          else bits[e] = (uint32_t)static_cast<const uint16_t*>(grad)[i0 + e] << 16;
        }
      }
    }
    if (mask != nullptr && cnt > 0) {
      const uint32_t m = (mask[i0 >> 5] >> (unsigned)(i0 & 31)) & 0xFu;
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (m & (1u << e)) bits[e] = 0;
    }
    return cnt;
  }

  // elements i0..i0+3 all exist (no bounds checks)
  __device__ __forceinline__ void load_full4(unsigned long long i0, uint32_t (&bits)[4]) const {
    if (DTYPE == NSML_F32) {
      const uint4 v = __ldcs(reinterpret_cast<const uint4*>(static_cast<const uint32_t*>(grad) + i0));
      bits[0] = v.x; bits[1] = v.y; bits[2] = v.z; bits[3] = v.w;
    } else {
      const uint2 v = __ldcs(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(grad) + i0));
      bits[0] = v.x << 16; bits[1] = v.x & 0xFFFF0000u;
      bits[2] = v.y << 16; bits[3] = v.y & 0xFFFF0000u;
    }
    if (mask != nullptr) {
      const uint32_t m = (mask[i0 >> 5] >> (unsigned)(i0 & 31)) & 0xFu;
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (m & (1u << e)) bits[e] = 0;
    }
  }

  // element i as stored (no pruning mask applied), and whether the mask prunes it
  __device__ __forceinline__ uint32_t raw1(unsigned long long i) const {
    if (DTYPE == NSML_F32) return static_cast<const uint32_t*>(grad)[i];
    return (uint32_t)static_cast<const uint16_t*>(grad)[i] << 16;
  }
  __device__ __forceinline__ bool pruned(unsigned long long i) const {
    return mask != nullptr && ((mask[i >> 5] >> (unsigned)(i & 31)) & 1u);
  }

  __device__ __forceinline__ uint32_t load1(unsigned long long i) const {
    if (mask != nullptr && ((mask[i >> 5] >> (unsigned)(i & 31)) & 1u)) return 0;
    if (DTYPE == NSML_F32) return static_cast<const uint32_t*>(grad)[i];
    return (uint32_t)static_cast<const uint16_t*>(grad)[i] << 16;
  }
};

}  // namespace nsml
