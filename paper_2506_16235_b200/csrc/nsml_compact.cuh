// Bucket -> candidate list: the one full pass over the bucket (Alg. 2 Steps 2-3:
// pruned gradients read as zero; everything whose magnitude is below the sampled
// lower bound is dropped here, in one streaming read).
//
// The bucket is cut into tiles of kTileBytes.  A block takes a tile and appends
// what it keeps (every key >= lo) to the tile's own slots of the list,
// [t * tile, t * tile + count), in index order, so nothing can overflow, nothing
// is allocated and no block ever waits for another; tiles in increasing order
// are in index order.  Keys inside the sampled window are counted in 4096 bins
// on the way (fire-and-forget reductions), so that the list stage knows the
// threshold's bin without a pass over the list.
#pragma once

#include "nsml_common.cuh"

namespace nsml {

// |v| >= t on floats equals key >= lo for finite v; written as !(|v| < t) so
// that NaN is kept too (k_emit reports non-finite candidates).
template <int EPL>
__device__ __forceinline__ unsigned int keep_flags(const uint32_t (&bits)[EPL], float t) {
  unsigned int f = 0;
#pragma unroll
  for (int e = 0; e < EPL; ++e) f |= (unsigned)(!(fabsf(__uint_as_float(bits[e])) < t)) << e;
  return f;
}

// One 16-byte load of a lane, unpacked: float32 as is, bfloat16 widened to float32 bit patterns.
template <int DTYPE, int EPL>
__device__ __forceinline__ void unpack16(const uint4& v, uint32_t (&bits)[EPL]) {
  if (DTYPE == NSML_F32) {
    bits[0] = v.x; bits[1] = v.y; bits[2] = v.z; bits[3] = v.w;
  } else {
    bits[0] = v.x << 16; bits[1] = v.x & 0xFFFF0000u;
    bits[2] = v.y << 16; bits[3] = v.y & 0xFFFF0000u;
    bits[4 % EPL] = v.z << 16; bits[5 % EPL] = v.z & 0xFFFF0000u;
    bits[6 % EPL] = v.w << 16; bits[7 % EPL] = v.w & 0xFFFF0000u;
  }
}

struct TileList {  // where the bucket pass leaves what it keeps
  unsigned short* off;        // see CompressLayout
  uint32_t* val;
  unsigned int* tile_count;
  unsigned int* group_count;
  unsigned int* window_hist;
  uint2* bins;                // (key, index) by bin of the window; not where a bin holds one key
  unsigned int bin_room;
  unsigned long long* chunk_sum[2];
  unsigned int* block_fill;
  unsigned int group_shift;
};

// Shared memory of a block of the bucket pass: what it keeps of its tile, in index order.
template <bool PACKED>
struct KeepShared {
  static constexpr int TILE = PACKED ? tile_elems<NSML_BF16>() : tile_elems<NSML_F32>();
  __align__(16) uint32_t val[TILE];
  __align__(8) unsigned short off[PACKED ? 4 : TILE];
  unsigned int cnt[kCta / 32];
  unsigned int few[kFewBins];
};

// Keeps a tile's candidates.  A warp's share of the tile is 4 rounds of 32 lanes x EPL elements, `first` = its offset
// in the tile, bits_of(r, bits) fetches a lane's EPL elements of round r.  PACKED: entries are offset << 16 | bfloat16
// bits.  The candidates are put in order in shared memory and then written, four per thread, in whole sectors; the
// window's histogram is counted on the way out, by full warps.  Reductions to one address run at about two per
// nanosecond, so adds must not pile up on a few of them: a window of few bins (bfloat16 keys: a window is a handful of
// key values) is counted in shared memory first, and in a tile that is full of candidates the lanes of a warp with
// equal bins add once.
template <int EPL, bool PACKED, class Bits>
__device__ __forceinline__ void keep_tile(const TileList& out, unsigned long long tile, unsigned int first, const Window& win,
                                          Ctl* ctl, KeepShared<PACKED>& sh, unsigned long long n, Bits&& bits_of) {
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned int lt = (1u << lane) - 1u;
  const float t = __uint_as_float(win.lo);
  unsigned int flags[4], mine = 0;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    uint32_t bits[EPL];
    bits_of(r, bits);
    flags[r] = keep_flags<EPL>(bits, t);
    if (win.lo == 0) {  // everything is kept: not what the bucket's ragged end is padded with
      const unsigned long long i = tile * (unsigned long long)KeepShared<PACKED>::TILE + first + (r * 32 + lane) * EPL;
      if (i + EPL > n) flags[r] &= i < n ? (1u << (n - i)) - 1u : 0u;
    }
    mine += __popc(flags[r]);
  }
  const unsigned int warp_total = __reduce_add_sync(FULL, mine);
  if (lane == 0) sh.cnt[warp] = warp_total;
  if (win.few && threadIdx.x < kFewBins) sh.few[threadIdx.x] = 0;
  __syncthreads();
  unsigned int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kCta / 32; ++w) {
    const unsigned int c = sh.cnt[w];
    if (w < warp) before += c;
    total += c;
  }
  if (threadIdx.x == 0) {
    out.tile_count[tile] = total;
    if (total) {
      if (out.group_shift == 0) out.group_count[tile] = total;
      else atomicAdd(out.group_count + (tile >> out.group_shift), total);
    }
  }
  constexpr int kChunksPerTile = KeepShared<PACKED>::TILE / kChunk;
  if (threadIdx.x < kChunksPerTile) {  // clear the list stage's counters on the way
    const unsigned long long c = tile * kChunksPerTile + threadIdx.x;
    out.chunk_sum[0][c] = 0;
    out.chunk_sum[1][c] = 0;
    out.block_fill[c] = 0;
  }
  if (total == 0) return;
  if (warp_total != 0) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const unsigned int f = flags[r];
      const unsigned int any = __ballot_sync(FULL, f != 0);
      if (any == 0) continue;
      unsigned int rank, round_total;
      if (__ballot_sync(FULL, (f & (f - 1)) != 0) == 0) {  // usual case: no lane keeps more than one element
        rank = __popc(any & lt);
        round_total = __popc(any);
      } else {
        const unsigned int cnt = __popc(f);
        unsigned int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned int up = __shfl_up_sync(FULL, incl, o);
          if (lane >= o) incl += up;
        }
        rank = incl - cnt;
        round_total = __shfl_sync(FULL, incl, 31);
      }
      uint32_t bits[EPL];
      bits_of(r, bits);
      unsigned int pos = before + rank;
#pragma unroll
      for (int e = 0; e < EPL; ++e) {
        if (f & (1u << e)) {
          const unsigned int off = first + r * 32 * EPL + lane * EPL + e;
          if (PACKED) {
            sh.val[pos] = off << 16 | bits[e] >> 16;
          } else {
            sh.val[pos] = bits[e];
            sh.off[pos] = (unsigned short)off;
          }
          ++pos;
        }
      }
      before += round_total;
    }
  }
  __syncthreads();
  const unsigned long long base = tile * (unsigned long long)KeepShared<PACKED>::TILE;
  const bool crowded = total > kCta * 4;
  for (unsigned int i0 = warp * 128; i0 < total; i0 += kCta * 4) {  // (uniform over the warp)
    const unsigned int i = i0 + lane * 4;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (i < total) {  // (up to three entries past the last one are copied too; the tile's slots have room)
      v = *reinterpret_cast<const uint4*>(sh.val + i);
      *reinterpret_cast<uint4*>(out.val + base + i) = v;
      if (!PACKED) *reinterpret_cast<uint2*>(out.off + base + i) = *reinterpret_cast<const uint2*>(sh.off + (PACKED ? 0 : i));
    }
    const uint32_t e4[4] = {v.x, v.y, v.z, v.w};
    uint32_t key[4];
    unsigned int bin[4], slot[4];
    bool inside[4], nonfinite = false;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      key[e] = (PACKED ? e4[e] << 16 : e4[e]) & 0x7FFFFFFFu;
      const bool live = i + e < total;
      nonfinite |= live && key[e] >= kInfKey;
      inside[e] = live && key[e] < win.hi;  // (key >= lo)
      bin[e] = (key[e] - win.lo) >> win.shift;
      slot[e] = 0;
    }
    if (nonfinite) set_status(&ctl->status, NSML_ERR_NONFINITE);
    if (crowded) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const unsigned int who = __ballot_sync(FULL, inside[e]);
        if (inside[e]) {
          const unsigned int same = __match_any_sync(who, bin[e]);
          const int leader = __ffs(same) - 1;
          unsigned int base_slot = 0;
          if (lane == leader) {
            if (win.few) atomicAdd(&sh.few[bin[e]], (unsigned int)__popc(same));
            else base_slot = atomicAdd(out.window_hist + bin[e], (unsigned int)__popc(same));
          }
          slot[e] = __shfl_sync(same, base_slot, leader) + __popc(same & lt);
        }
      }
    } else if (win.few) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (inside[e]) atomicAdd(&sh.few[bin[e]], 1u);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)  // (the four are in flight together)
        if (inside[e]) slot[e] = atomicAdd(out.window_hist + bin[e], 1u);
    }
    if (!win.single()) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (inside[e] && slot[e] < out.bin_room)
          out.bins[(size_t)bin[e] * out.bin_room + slot[e]] = make_uint2(key[e], (uint32_t)base + (PACKED ? e4[e] >> 16 : sh.off[PACKED ? 0 : i + e]));
    }
  }
  if (win.few) {
    __syncthreads();
    if (threadIdx.x < kFewBins) {
      const unsigned int c = sh.few[threadIdx.x];
      if (c) atomicAdd(out.window_hist + threadIdx.x, c);
    }
  }
}

// The bucket pass is NOT a persistent kernel.  A block is eight warps on one tile (16 consecutive KB); a warp issues
// all of its loads at once and is done.  The hardware's block scheduler, which hands out blocks in order, keeps the
// grid on one compact, moving window of the bucket.  Measured on a 100 MB float32 bucket whose candidates crowd into
// a few tensors: 19.0 us, against 19.9 us for persistent blocks that prefetch the next segment into registers, 21.9 us
// for a shared-memory ring of asynchronous copies and 18.6 us for a plain read of the bucket; blocks that own 2, 4, 8
// consecutive 16 KB steps take 20.5, 23.4, 29.4 us (the wider the window of addresses in flight, the slower).
// Short-lived blocks also share the SMs gracefully with other streams' kernels.  The first wave's loads are issued
// while the sample kernel still runs.
//
// FEEDBACK: the bucket that is compressed is gradient + residual (Section 4.2 Step 3, local accumulation of the
// filtered gradients).  The residual is streamed beside the gradient, the sum (one float32 add per element) is
// written back over the residual and is what the candidates are taken from; the pruning mask zeroes a key, not the
// stored sum.  A tile is then 4096 sums whatever the gradient's type.
// MASKED: a pruning mask is applied (a warp's mask words are fetched with the data and handed out by shuffle).
template <int DTYPE, bool FEEDBACK, bool MASKED>
__global__ void __launch_bounds__(kCta, FEEDBACK ? 4 : 5)
k_compact_bucket(BucketSrc<DTYPE> src, float* __restrict__ residual, unsigned long long n, Ctl* ctl, TileList out) {
  __shared__ KeepShared<!FEEDBACK && DTYPE == NSML_BF16> sh;
  constexpr int ESIZE = (DTYPE == NSML_F32) ? 4 : 2;
  constexpr int EPL = FEEDBACK ? 4 : 16 / ESIZE;  // elements a lane takes per round
  constexpr int ROUND = 32 * EPL;                 // elements a warp handles per round
  constexpr int SHARE = 4 * ROUND;                // elements of a warp: 512 or 1024
  constexpr unsigned long long TILE = FEEDBACK ? tile_elems<NSML_F32>() : tile_elems<DTYPE>();
  static_assert(SHARE * (kCta / 32) == TILE, "a block is a tile");
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned long long tile = blockIdx.x;
  const unsigned int first = warp * SHARE;
  const unsigned long long i0 = tile * TILE + first;  // the warp's first element
  uint4 q[4];  // the lane's elements: as loaded, or (FEEDBACK) the sums
  float4 res[FEEDBACK ? 4 : 1];
  const bool whole = i0 + SHARE <= n;
  if (whole) {
    const unsigned char* g = static_cast<const unsigned char*>(src.grad) + (i0 + lane * EPL) * ESIZE;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (EPL * ESIZE == 16) {
        q[r] = __ldcs(reinterpret_cast<const uint4*>(g + r * ROUND * ESIZE));
      } else {  // four bfloat16
        const uint2 v = __ldcs(reinterpret_cast<const uint2*>(g + r * ROUND * ESIZE));
        q[r] = make_uint4(v.x, v.y, 0u, 0u);
      }
    }
    if (FEEDBACK) {
#pragma unroll
      for (int r = 0; r < 4; ++r) res[FEEDBACK ? r : 0] = __ldcs(reinterpret_cast<const float4*>(residual + i0 + r * ROUND + lane * EPL));
    }
  }
  uint32_t mw = 0;
  if (MASKED && lane < SHARE / 32 && i0 + lane * 32ull < n) mw = __ldg(src.mask + i0 / 32 + lane);
  if (FEEDBACK && whole) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      uint32_t b[4];
      if (DTYPE == NSML_F32) {
        b[0] = q[r].x; b[1] = q[r].y; b[2] = q[r].z; b[3] = q[r].w;
      } else {
        b[0] = q[r].x << 16; b[1] = q[r].x & 0xFFFF0000u;
        b[2] = q[r].y << 16; b[3] = q[r].y & 0xFFFF0000u;
      }
      const float4 a = res[FEEDBACK ? r : 0];
      const float4 sum = make_float4(__fadd_rn(__uint_as_float(b[0]), a.x), __fadd_rn(__uint_as_float(b[1]), a.y),
                                     __fadd_rn(__uint_as_float(b[2]), a.z), __fadd_rn(__uint_as_float(b[3]), a.w));
      q[r] = make_uint4(__float_as_uint(sum.x), __float_as_uint(sum.y), __float_as_uint(sum.z), __float_as_uint(sum.w));
    }
  }
  pdl_wait();
  if (FEEDBACK && whole) {
#pragma unroll
    for (int r = 0; r < 4; ++r) *reinterpret_cast<uint4*>(residual + i0 + r * ROUND + lane * EPL) = q[r];
  }
  if (!whole) {
    // the bucket's ragged end: plain loads, missing elements read as 0 and are never kept
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int e = 0; e < EPL; ++e) {
        const unsigned long long i = i0 + r * ROUND + lane * EPL + e;
        if (i >= n) continue;
        if (FEEDBACK) {
          const float sum = __fadd_rn(__uint_as_float(src.raw1(i)), residual[i]);
          residual[i] = sum;
          w[e & 3] = __float_as_uint(sum);
        } else if (DTYPE == NSML_F32) {
          w[e & 3] = src.raw1(i);
        } else {
          w[(e >> 1) & 3] |= (src.raw1(i) >> 16) << (16 * (e & 1));
        }
      }
      q[r] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  const Window win = make_window<FEEDBACK ? NSML_F32 : DTYPE>(ctl);
  keep_tile<EPL, !FEEDBACK && DTYPE == NSML_BF16>(out, tile, first, win, ctl, sh, n, [&](int r, uint32_t (&bits)[EPL]) {
    unpack16<FEEDBACK ? NSML_F32 : DTYPE, EPL>(q[r], bits);
    if (MASKED) {
      // this lane's EPL mask bits inside the round's ROUND / 32 words
      const uint32_t word = __shfl_sync(0xFFFFFFFFu, mw, r * (ROUND / 32) + lane * EPL / 32);
      const uint32_t m = (word >> (unsigned)((lane * EPL) & 31)) & ((1u << EPL) - 1u);
#pragma unroll
      for (int e = 0; e < EPL; ++e)
        if (m & (1u << e)) bits[e] = 0;
    }
  });
}

}  // namespace nsml
