// Sampled bounds of the top-k threshold (Alg. 2 Step 3: which k = ceil(ratio*n)
// gradients have the largest absolute value).
//
// The bucket is streamed exactly once, by the compaction pass, which needs a
// key `lo` such that a little more than k keys are >= lo, and counts the keys
// between lo and a second bound `hi` that a little fewer than k keys exceed.
// k_sample reads 16 bytes (4 float32 or 8 bfloat16 keys) from each of 16384 equal
// strata of the bucket and takes the two sample keys whose ranks lie six standard
// deviations either side of the expected rank of the k-th largest, rounded
// outwards to their top 14 bits.  (The keys of a stratum lie side by side; where
// neighbours are alike, as in the rows of a sparse embedding gradient, they count
// for less than as many independent draws, in the extreme case for one.)  The exact threshold is found
// afterwards (nsml_list.cuh), which also repairs the rare case of a misleading
// sample, so the sample only decides how much work is done, never the result.
//
// What bounds the kernel is latency: launch, one round of scattered reads, the
// select.  It is one cluster of eight blocks; a block counts its keys' top 14
// bits in shared memory, then sums an eighth of
// the bins over the eight blocks through distributed shared memory, so that one
// counting level and two cluster barriers replace the two levels in a single
// block that an exact 24-bit select takes.
#pragma once

#include <cooperative_groups.h>

#include "nsml_common.cuh"

namespace nsml {

constexpr int kSampleThreads = 1024;
constexpr int kSampleBlocks = 8;
constexpr int kSampleLoads = 2;  // strata per thread
static_assert(kSamples == kSampleThreads * kSampleBlocks * kSampleLoads, "every stratum has a thread");

__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x ^= x >> 16; x *= 0x7FEB352Du;
  x ^= x >> 15; x *= 0x846CA68Bu;
  x ^= x >> 16;
  return x;
}

// Block-wide search from the top over bins held PER per thread (own[] holds
// this thread's consecutive bins, lowest first): leaves in s_out the digit d
// with #{digit > d} < rem <= #{digit >= d}, the rank left inside bin d and the bin's count.
// Called by every thread of the block; s_tot needs one word per warp.
template <int PER, int THREADS>
__device__ __forceinline__ void find_digit_from_top(const unsigned int (&own)[PER], unsigned int rem,
                                                    unsigned int* s_tot, unsigned int* s_out) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  unsigned int mine = 0;
#pragma unroll
  for (int b = 0; b < PER; ++b) mine += own[b];
  unsigned int incl = mine;  // this thread and all higher lanes of the warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int v = __shfl_down_sync(0xFFFFFFFFu, incl, o);
    if (lane + o < 32) incl += v;
  }
  __syncthreads();  // s_tot and s_out may still be read from an earlier call
  if (lane == 0) s_tot[warp] = incl;
  __syncthreads();
  static_assert(THREADS <= 1024, "a warp's lanes hold all warps' counts");
  unsigned int above = incl - mine + __reduce_add_sync(0xFFFFFFFFu, lane > warp && lane < THREADS / 32 ? s_tot[lane] : 0u);
  if (above < rem && rem <= above + mine) {  // exactly one thread
#pragma unroll
    for (int b = PER - 1; b >= 0; --b) {
      if (rem <= above + own[b]) {
        s_out[0] = (unsigned)(t * PER + b);
        s_out[1] = rem - above;
        s_out[2] = own[b];
        break;
      }
      above += own[b];
    }
  }
  __syncthreads();
}

// Keys are counted by their top 14 bits (64 bins per octave) over the 108 octaves from 2^-76 to 2^32, by their top 11 bits
// below and above, in 16-bit counters: 16 KB that eight blocks read from one another.  (All of the top 15 bits, 64 KB: the
// sum over the blocks took 3 us, now 1.  With 128 octaves from 2^-96 on and nothing below, buckets around 1e-30 at 0.01
// had no lower bound, so that all of them were listed: 16M float32 elements 3120 us, now 53,
// where an ordinary call takes 47.)
constexpr int kSampleShift = 17, kSampleCoarse = 3;  // a fine bin is 2^17 keys, a coarse one 2^20
constexpr unsigned int kSampleBins = 8192;
constexpr unsigned int kSampleFine = 51u << 6, kSampleAbove = 159u << 6;  // key >> 17 of the first fine one, and behind the last
constexpr unsigned int kSampleFineBin = kSampleFine >> kSampleCoarse;     // their bins
constexpr unsigned int kSampleAboveBin = kSampleFineBin + kSampleAbove - kSampleFine;
static_assert(kSampleAboveBin + ((1u << 14) - kSampleAbove >> kSampleCoarse) <= kSampleBins, "every key has a bin");
__device__ __forceinline__ unsigned int sample_bin(uint32_t key) {  // 0: not counted
  const int at = (int)(key >> kSampleShift), fine = min(max(at, (int)kSampleFine), (int)kSampleAbove);
  return ((at - fine) >> kSampleCoarse) + fine + (int)kSampleFineBin - (int)kSampleFine;  // (a select per range: 0.3 us more)
}
__device__ __forceinline__ uint32_t sample_bin_begin(unsigned int bin) {  // (behind the last bin: 0x80000000)
  if (bin < kSampleFineBin) return bin << (kSampleShift + kSampleCoarse);
  if (bin < kSampleAboveBin) return (bin - kSampleFineBin + kSampleFine) << kSampleShift;
  return (((bin - kSampleAboveBin) << kSampleCoarse) + kSampleAbove) << kSampleShift;
}
__device__ __forceinline__ uint32_t sample_bin_end(unsigned int bin) { return sample_bin_begin(bin + 1); }

// Clears the per-call control region and sets ctl->lo and ctl->hi from a stratified sample of the bucket (of
// bucket + addend when an addend is given).  rank_lo, rank_hi: ranks from the top among the sampled keys.  A rank
// beyond the non-zero sample keys leaves its bound 0.
template <int DTYPE>
__global__ void __cluster_dims__(kSampleBlocks, 1, 1) __launch_bounds__(kSampleThreads)
k_sample(BucketSrc<DTYPE> src, const float* __restrict__ addend, unsigned long long n, unsigned int rank_lo, unsigned int rank_hi,
         Ctl* ctl, uint4* zero_base, unsigned int zero_vec16, int keep_status) {
  namespace cg = cooperative_groups;
  constexpr int KEYS = sample_keys<DTYPE>();
  __shared__ __align__(16) unsigned int s_bins[kSampleBins / 2];  // two 16-bit counters per word
  __shared__ unsigned int s_scan[kSampleThreads / 32];
  __shared__ unsigned int s_slice[kSampleBlocks];  // keys in each block's slice of the bins
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned int rank = cluster.block_rank();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  static_assert(kSampleBins / 8 == kSampleThreads, "eight counters per thread");
  reinterpret_cast<uint4*>(s_bins)[t] = make_uint4(0u, 0u, 0u, 0u);
  pdl_wait();

  uint4 raw[kSampleLoads];
  float add[kSampleLoads][KEYS];
  uint32_t pruned[kSampleLoads];  // bit e: key e of the stratum is pruned
#pragma unroll
  for (int s = 0; s < kSampleLoads; ++s) {
    const unsigned long long stratum = ((unsigned long long)s * kSampleBlocks + rank) * kSampleThreads + t;
    const unsigned long long begin = stratum * n / kSamples;
    const unsigned long long end = (stratum + 1) * n / kSamples;  // > begin
    unsigned long long pos = (begin + mix32((uint32_t)stratum * 0x9E3779B1u + 0x85EBCA6Bu) % (uint32_t)(end - begin)) & ~(unsigned long long)(KEYS - 1);
    if (pos + KEYS > n) pos = (n - KEYS) & ~(unsigned long long)(KEYS - 1);  // (n >= KEYS)
    raw[s] = __ldcs(reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(src.grad) + pos * (DTYPE == NSML_F32 ? 4 : 2)));
#pragma unroll
    for (int e = 0; e < KEYS; e += 4) {
      const float4 a = addend != nullptr ? *reinterpret_cast<const float4*>(addend + pos + e) : make_float4(0.f, 0.f, 0.f, 0.f);
      add[s][e] = a.x; add[s][e + 1] = a.y; add[s][e + 2] = a.z; add[s][e + 3] = a.w;
    }
    pruned[s] = src.mask != nullptr ? __ldg(src.mask + (pos >> 5)) >> (unsigned)(pos & 31) : 0u;
  }
  // keep_status: an error an earlier step of the same call left in the status word stays visible
  for (unsigned int i = rank * kSampleThreads + t; i < zero_vec16; i += kSampleBlocks * kSampleThreads)
    zero_base[i] = make_uint4((i == 0 && keep_status) ? (unsigned int)ctl->status : 0u, 0, 0, 0);
  __syncthreads();
  unsigned int low_bits = 0;
#pragma unroll
  for (int s = 0; s < kSampleLoads; ++s) {
    uint32_t bits[KEYS];
    if (DTYPE == NSML_F32) {
      bits[0] = raw[s].x; bits[1] = raw[s].y; bits[2] = raw[s].z; bits[3] = raw[s].w;
    } else {
      bits[0] = raw[s].x << 16; bits[1] = raw[s].x & 0xFFFF0000u;
      bits[2] = raw[s].y << 16; bits[3] = raw[s].y & 0xFFFF0000u;
      bits[4 % KEYS] = raw[s].z << 16; bits[5 % KEYS] = raw[s].z & 0xFFFF0000u;
      bits[6 % KEYS] = raw[s].w << 16; bits[7 % KEYS] = raw[s].w & 0xFFFF0000u;
    }
#pragma unroll
    for (int e = 0; e < KEYS; ++e) {
      // with an addend (the residual of the local accumulation) the bucket that is selected from is the sum
      if (addend != nullptr) bits[e] = __float_as_uint(__fadd_rn(__uint_as_float(bits[e]), add[s][e]));
      if ((pruned[s] >> e) & 1u) bits[e] = 0;
      low_bits |= bits[e] & 0xFFFFu;
      const unsigned int bin = sample_bin(bits[e] & 0x7FFFFFFFu);
      if (bin != 0) atomicAdd(&s_bins[bin >> 1], 1u << (16 * (bin & 1)));  // (a block has at most 16384 keys: no overflow)
    }
  }
  // The bucket pass may start to load: only now, when what the stream did before this kernel is complete, and behind
  // this kernel's own reads.
  pdl_launch_dependents();
  // (a float32 key has its low 13 bits zero once in 8192; a few odd keys do not matter here)
  const int below16 = DTYPE == NSML_F32 && addend == nullptr ? __syncthreads_count(low_bits != 0) : kSampleThreads;
  const int below13 = DTYPE == NSML_F32 && addend == nullptr ? __syncthreads_count((low_bits & 0x1FFFu) != 0) : kSampleThreads;
  cluster.sync();  // every block's counts are complete, the control region is cleared
  if (rank == 0 && t == 0) ctl->grain = below16 < kSampleThreads / 16 ? 16 : below13 < kSampleThreads / 16 ? 13 : 0;

  // this block's slice of the bins, two per thread of the lower half, summed over the blocks
  constexpr unsigned int kSlice = kSampleBins / kSampleBlocks;
  static_assert(kSlice == kSampleThreads, "a word of two bins for every other thread");
  unsigned int own[2] = {0, 0};
  if (t < (int)kSlice / 2) {
    unsigned int v[kSampleBlocks];
#pragma unroll
    for (int b = 0; b < kSampleBlocks; ++b) v[b] = cluster.map_shared_rank(s_bins, b)[rank * (kSlice / 2) + t];
#pragma unroll
    for (int b = 0; b < kSampleBlocks; ++b) {
      own[0] += v[b] & 0xFFFFu;
      own[1] += v[b] >> 16;
    }
  }
  const unsigned int mine = own[0] + own[1];
  unsigned int incl = mine;  // this thread and all higher lanes of the warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int v = __shfl_down_sync(0xFFFFFFFFu, incl, o);
    if (lane + o < 32) incl += v;
  }
  if (lane == 0) s_scan[warp] = incl;
  __syncthreads();
  const unsigned int of_warp = s_scan[lane], total = __reduce_add_sync(0xFFFFFFFFu, of_warp);
  unsigned int above = incl - mine + __reduce_add_sync(0xFFFFFFFFu, lane > warp ? of_warp : 0u);
  if (t < kSampleBlocks) *cluster.map_shared_rank(&s_slice[rank], t) = total;
  cluster.sync();  // also: no block leaves while its bins are still read
  for (int s = rank + 1; s < kSampleBlocks; ++s) above += s_slice[s];
#pragma unroll
  for (int which = 0; which < 2; ++which) {
    const unsigned int j = which == 0 ? rank_lo : rank_hi;
    if (above < j && j <= above + mine) {  // exactly one thread of the cluster, if any
      unsigned int a = above;
#pragma unroll
      for (int b = 1; b >= 0; --b) {
        if (a < j && j <= a + own[b]) {
          const unsigned int bin = rank * kSlice + t * 2 + b;
          if (which == 0) ctl->lo = sample_bin_begin(bin);
          else ctl->hi = sample_bin_end(bin);
        }
        a += own[b];
      }
    }
  }
}

}  // namespace nsml
