// The steps of Alg. 2 around the top-k selection:
//   Step 1  the gradient's L2 norm for the adaptive-quantisation gate (k_sumsq)
//   Step 2  the pruning mask built from the weights: the ceil(0.5*(1-ratio)*n)
//           parameters of smallest magnitude, ties by lower index
//           (k_sample, k_prune_pass, k_prune_finish)
// (Step 3, "accumulate the local filtered gradients", is part of the compress
// kernels: the bucket is gradient + residual, and the residual keeps what the
// payload does not carry.)
// The streaming kernels read with 16-byte loads on one moving window of memory:
// k_sumsq as one wave of blocks that take tiles block-cyclically, k_prune_pass
// with a short-lived block per tile.
#pragma once

#include "nsml_accumulate.cuh"
#include "nsml_list.cuh"

namespace nsml {

constexpr int kStreamLoads = 4;  // 16-byte loads a thread keeps in flight
constexpr int kStreamTile = kCta * 4 * kStreamLoads;  // elements a block takes per step

// ------------------------------------------------------------------------
// Step 1: sum of squares in float64.  Every square is exact in float64 (a
// float32 has 24 significant bits), the adds follow a fixed order for a given
// grid (per thread, per warp, per block, then the last block to finish adds
// the per-block sums in block order), so the result is reproducible.  A caller
// that waits for the sum gets it written to page-locked host memory (a copy to
// pageable memory behind the kernel took 6 us longer).
// ------------------------------------------------------------------------
struct SumsqCtl {
  int status;
  unsigned int ticket;  // blocks that have delivered their partial sum
  double sumsq;
};
constexpr int kSumsqMaxBlocks = 4096;
constexpr size_t kSumsqWorkspace = 256 + (size_t)kSumsqMaxBlocks * 8;

__device__ __forceinline__ double block_sum_f64(double t, double* s_red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = t;
  __syncthreads();
  double b = 0.0;
#pragma unroll
  for (int w = 0; w < kCta / 32; ++w) b += s_red[w];
  return b;
}

template <int DTYPE>
__global__ void __launch_bounds__(kCta)
k_sumsq(BucketSrc<DTYPE> src, unsigned long long n, SumsqCtl* ctl, double* __restrict__ partials, SumsqCtl* to_host) {
  __shared__ double s_red[kCta / 32];
  __shared__ unsigned int s_last;
  const unsigned long long tiles = (n + kStreamTile - 1) / kStreamTile;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  uint32_t worst = 0;  // largest magnitude key seen
  for (unsigned long long tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const unsigned long long base = tile * kStreamTile;
    uint32_t bits[kStreamLoads][4];
    if (base + kStreamTile <= n) {
#pragma unroll
      for (int u = 0; u < kStreamLoads; ++u) src.load_full4(base + (unsigned long long)(u * kCta + threadIdx.x) * 4, bits[u]);
    } else {
#pragma unroll
      for (int u = 0; u < kStreamLoads; ++u) src.load_vals4(base + (unsigned long long)(u * kCta + threadIdx.x) * 4, n, bits[u]);
    }
#pragma unroll
    for (int u = 0; u < kStreamLoads; ++u) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const double v = (double)__uint_as_float(bits[u][e]);
        acc[u & 3] = fma(v, v, acc[u & 3]);  // the product is exact, so this is one rounding, of the add
        worst = max(worst, bits[u][e] & 0x7FFFFFFFu);
      }
    }
  }
  if (worst >= kInfKey) set_status(&ctl->status, NSML_ERR_NONFINITE);
  const double block_total = block_sum_f64((acc[0] + acc[1]) + (acc[2] + acc[3]), s_red);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = block_total;
    __threadfence();
    s_last = atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();  // the other blocks' partial sums are visible
  double p = 0.0;
  for (unsigned int i = threadIdx.x; i < gridDim.x; i += kCta) p += __ldcg(partials + i);
  const double total = block_sum_f64(p, s_red);
  if (threadIdx.x == 0) {
    ctl->sumsq = total;
    ctl->ticket = 0;
    if (to_host != nullptr) {
      to_host->sumsq = total;
      to_host->status = __ldcg(&ctl->status);
    }
  }
}

// ------------------------------------------------------------------------
// Step 2: pruning mask from the weights: the m parameters of smallest magnitude,
// ties by lower index, in one pass over the weights.  A stratified sample
// (k_sample) brackets the m-th smallest magnitude; the pass (k_prune_pass) sets
// the bits of everything below the bracket and lists the weights inside it (about
// 3 % of them); k_prune_finish counts the listed keys in 4096 bins (and a large
// bin's keys in 4096 more), sets the bits
// of those below the threshold's bin, ranks that bin's few hundred keys
// (magnitude, then index) and sets the bits of the first of them.  When the
// sample misleads, the list is full, or the bin holds too many keys (massive
// ties), the same kernel does a radix select over the weights instead (12 + 12 +
// 7 bits, then the ties by their rank): the result is exact either way.
//
// Measured (24.4M weights): 11 + 34 + 18 us (sample, pass, finish), less what they
// overlap; before, eleven launches, 102 us: two passes over the weights (35 and 25
// us), a sample in one block (14), six kernels of the fallback that left at once (17).
// ------------------------------------------------------------------------
constexpr int kPruneTile = kCta * 16;       // weights per block of the pass
constexpr int kPruneThreads = 512;
constexpr unsigned int kPruneUnit = 8192;   // weights, or listed keys, per unit of work of k_prune_finish
constexpr unsigned int kTieCap = 1024;      // keys of the threshold's bin that are ranked

struct PruneLayout {
  size_t hist;       // u32[5][kMaxBins]: digits of the radix select; the last two count listed keys
  size_t zero_bytes; // everything before this offset is cleared per call
  size_t bin_list;   // uint2[kTieCap]: (key, index) of the threshold's bin
  size_t unit_ties;  // u32[units]: weights that tie with the threshold
  size_t list;       // uint2[cap]: (key, index) of the weights inside the bracket
  size_t cap, total;
};

inline PruneLayout prune_layout(int64_t n) {
  PruneLayout L;
  L.hist = 256;
  L.zero_bytes = L.hist + 5 * kMaxBins * sizeof(unsigned int);
  L.bin_list = L.zero_bytes;
  L.unit_ties = L.bin_list + kTieCap * sizeof(uint2);
  L.list = L.unit_ties + align_up(((size_t)n + kPruneUnit - 1) / kPruneUnit * 4, 256);
  L.cap = (size_t)n / 8 + 1024;
  L.total = L.list + align_up(L.cap * sizeof(uint2), 256);
  return L;
}

// A block per 4096 weights, all loads issued at once (short-lived blocks on one moving window read fastest).  Bound by
// instructions once the loads are in flight: two compares with two flag updates and one add per weight, the mask words by
// a three-step exchange among eight lanes, places in the list by one shared and one global add per warp and block (the
// list has no order).  A block spends most of its life waiting, for its loads and for its place in the list, so eight of them
// per SM (32 registers) are better than six: Alg. 2 on 24.4M weights 139.9 -> 137.1 us.
__global__ void __launch_bounds__(kCta, 8)
k_prune_pass(BucketSrc<NSML_F32> src, unsigned long long n, Ctl* ctl, uint2* __restrict__ list, unsigned int cap, uint32_t* __restrict__ mask) {
  __shared__ unsigned int s_count, s_base;  // count: below the bracket << 16 | inside it
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned long long i0 = (unsigned long long)blockIdx.x * kPruneTile + warp * 512;  // the warp's 512 weights
  uint32_t b[4][4];
  const bool whole = i0 + 512 <= n;
  if (whole) {
#pragma unroll
    for (int r = 0; r < 4; ++r) src.load_full4(i0 + r * 128 + lane * 4, b[r]);
  }
  if (threadIdx.x == 0) s_count = 0;
  __syncthreads();
  pdl_wait();
  if (!whole) {
#pragma unroll
    for (int r = 0; r < 4; ++r) src.load_vals4(i0 + r * 128 + lane * 4, n, b[r]);
  }
  const unsigned int lo = ctl->lo, hi = ctl->hi > lo ? ctl->hi : 0x80000000u;
  // (on the weight itself: key < E  <=>  |w| < float(E); NaN is not below anything)
  const float t_lo = __uint_as_float(min(lo, kInfKey)), t_hi = __uint_as_float(min(hi, kInfKey));
  unsigned int under = 0, inside = 0;  // bit r * 4 + e
  float bad = 0.f;                     // becomes NaN with the first weight that is not finite
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float w = __uint_as_float(b[r][e]);
      if (fabsf(w) < t_lo) under |= 1u << (r * 4 + e);
      if (fabsf(w) < t_hi) inside |= 1u << (r * 4 + e);
      bad = __fmaf_rn(w, 0.f, bad);
    }
  inside &= ~under;
  if (!(bad == 0.f)) set_status(&ctl->status, NSML_ERR_NONFINITE);
  if (!whole) {  // missing weights were read as 0
    unsigned int here = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const unsigned long long i = i0 + r * 128 + lane * 4;
      here |= (i + 4 <= n ? 15u : i < n ? (1u << (n - i)) - 1u : 0u) << (r * 4);
    }
    under &= here;
    inside &= here;
  }
  const unsigned int mine = __popc(inside);
  unsigned int count = (unsigned int)__popc(under) << 16 | mine, incl = count;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int up = __shfl_up_sync(FULL, incl, o);
    if (lane >= o) incl += up;
  }
  unsigned int at = 0;
  if (lane == 31 && incl != 0) at = atomicAdd(&s_count, incl);  // (at most 4096 of either kind: the halves do not meet)
  // A mask word is the nibbles of eight neighbouring lanes.  Each step hands half of the rounds to a partner and
  // doubles what is held of the others: 4 rounds of 4 bits, 2 of 8, 1 of 16, 1 of 32.
  {
    const bool odd = lane & 1, odd2 = lane & 2;
    const unsigned int give = odd ? under & 0xFFu : under >> 8, got = __shfl_xor_sync(FULL, give, 1);
    const unsigned int keep = odd ? under >> 8 : under;  // rounds 2, 3 in odd lanes, 0, 1 in even ones
    const unsigned int low = odd ? got : keep, high = odd ? keep : got;
    const unsigned int two = (low & 15u) | (high & 15u) << 4 | (low & 0xF0u) << 4 | (high & 0xF0u) << 8;
    const unsigned int got2 = __shfl_xor_sync(FULL, odd2 ? two & 0xFFu : two >> 8, 2), keep2 = (odd2 ? two >> 8 : two) & 0xFFu;
    const unsigned int one = odd2 ? got2 | keep2 << 8 : keep2 | got2 << 8;
    const unsigned int word = one | __shfl_down_sync(FULL, one, 4) << 16;
    const unsigned long long at_word = i0 / 32 + (((lane & 1) << 1) | (lane >> 1 & 1)) * 4 + (lane >> 3);
    if ((lane & 4) == 0 && at_word < (n + 31) / 32) mask[at_word] = word;
  }
  __syncthreads();
  const unsigned int all = s_count;
  if (threadIdx.x == 0 && all != 0)
    s_base = (unsigned int)atomicAdd(&ctl->below_listed, (unsigned long long)(all >> 16) << 32 | (all & 0xFFFFu));
  if ((all & 0xFFFFu) == 0) return;
  __syncthreads();
  at = s_base + (__shfl_sync(FULL, at, 31) & 0xFFFFu) + ((incl - count) & 0xFFFFu);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    if ((inside >> (r * 4) & 15u) == 0) continue;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (inside & (1u << (r * 4 + e))) {
        if (at < cap) list[at] = make_uint2(b[r][e] & 0x7FFFFFFFu, (uint32_t)i0 + r * 128 + lane * 4 + e);
        ++at;
      }
  }
}

struct PruneShared {
  unsigned int hist[kMaxBins], tot[kPruneThreads / 32], out[3], ticket[2], done[2];
  unsigned int warp_ties[kPruneThreads / 32];
  uint2 bin[kTieCap];
};

__global__ void __launch_bounds__(kPruneThreads, 2)
k_prune_finish(BucketSrc<NSML_F32> src, unsigned int n, unsigned int m, Ctl* ctl, unsigned int* __restrict__ ghist, const uint2* __restrict__ list,
               unsigned int cap, uint2* __restrict__ bin_list, unsigned int* __restrict__ unit_ties, uint32_t* __restrict__ mask, int sampled) {
  constexpr int THREADS = kPruneThreads, NW = THREADS / 32, PER = kMaxBins / THREADS;
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  __shared__ PruneShared sh;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned int lt = (1u << lane) - 1u;
  pdl_wait();
  pdl_launch_dependents();
  auto clear = [&] {
    __syncthreads();
    for (int b = t; b < kMaxBins; b += THREADS) sh.hist[b] = 0;
  };
  auto flush = [&](unsigned int* to) {
    for (int b = t; b < kMaxBins; b += THREADS)
      if (sh.hist[b]) atomicAdd(to + b, sh.hist[b]);
  };
  // finds the bin that holds the rem-th largest counted key: sh.out
  auto find = [&](const unsigned int* from, unsigned int rem) {
    unsigned int own[PER];
#pragma unroll
    for (int b = 0; b < PER; ++b) own[b] = __ldcg(from + t * PER + b);
    find_digit_from_top<PER, THREADS>(own, rem, sh.tot, sh.out);
  };

  const unsigned int below = (unsigned int)(ctl->below_listed >> 32), listed = (unsigned int)ctl->below_listed;
  if (sampled && listed <= cap && below < m && m <= below + listed) {  // uniform over the grid
    const unsigned int lo = ctl->lo, hi = ctl->hi > lo ? ctl->hi : 0x80000000u;
    const unsigned int units = (listed + kPruneUnit / 4 - 1) / (kPruneUnit / 4);
    // the bin [first, first + width) of the threshold, which is the rem-th largest of its in_bin keys
    unsigned int first = lo, width = hi - lo, in_bin = listed, rem = listed - (m - below) + 1;
    for (int level = 0; level < 2 && in_bin > kTieCap && width > 1; ++level) {
      const unsigned int span = (width - 1) / kMaxBins, shift = span == 0 ? 0u : 32u - __clz(span);
      clear();
      if (!run_phase(ctl, level, units, sh, [&](unsigned int u) {
#pragma unroll
            for (unsigned int q = 0; q < kPruneUnit / 4 / THREADS; ++q) {
              const unsigned int i = u * (kPruneUnit / 4) + q * THREADS + t;
              const unsigned int rel = i < listed ? __ldcg(&list[i].x) - first : FULL;
              if (rel < width) atomicAdd(&sh.hist[rel >> shift], 1u);
            }
          }, [&] { flush(ghist + (3 + level) * kMaxBins); }))
        return;
      find(ghist + (3 + level) * kMaxBins, rem);
      first += sh.out[0] << shift;
      width = 1u << shift;
      rem = sh.out[1];
      in_bin = sh.out[2];
    }
    const unsigned int take = in_bin - rem + 1;  // the bin's smallest `take` keys are pruned
    if (in_bin <= kTieCap) {
      const bool ok = run_phase(ctl, 2, units, sh, [&](unsigned int u) {
#pragma unroll
        for (unsigned int q = 0; q < kPruneUnit / 4 / THREADS; ++q) {
          const unsigned int i = u * (kPruneUnit / 4) + q * THREADS + t;
          if (i >= listed) continue;
          const uint2 e = __ldcg(list + i);
          if (e.x < first) {
            atomicOr(mask + (e.y >> 5), 1u << (e.y & 31));
          } else if (e.x - first < width) {
            const unsigned int slot = atomicAdd(&ctl->done, 1u);
            if (slot < kTieCap) bin_list[slot] = e;
          }
        }
      }, [] {});
      if (!ok) return;
      // a warp per key of the bin, the lanes share the comparisons
      for (unsigned int i = t; i < in_bin; i += THREADS) sh.bin[i] = __ldcg(bin_list + i);
      __syncthreads();
      for (unsigned int i = blockIdx.x * NW + warp; i < in_bin; i += gridDim.x * NW) {
        const uint2 me = sh.bin[i];
        unsigned int before = 0;
        for (unsigned int q = lane; q < in_bin; q += 32) {
          const uint2 e = sh.bin[q];
          before += e.x < me.x || (e.x == me.x && e.y < me.y);
        }
        before = __reduce_add_sync(FULL, before);
        if (lane == 0 && before < take) atomicOr(mask + (me.y >> 5), 1u << (me.y & 31));
      }
      return;
    }
  }

  // ---------------- radix select over the weights ----------------
  const unsigned int units = (n + kPruneUnit - 1) / kPruneUnit;
  unsigned int prefix = 0, rem = n - m + 1;  // the threshold is the rem-th largest magnitude
  for (int level = 0; level < 3; ++level) {
    const int shift = digit_shift(level), above = level == 0 ? 31 : digit_shift(level - 1);
    const unsigned int digit_mask = (1u << digit_bits(level)) - 1u;
    bool nonfinite = false;
    clear();
    const bool ok = run_phase(ctl, 3 + level, units, sh, [&](unsigned int u) {
      for (unsigned int q = 0; q < kPruneUnit / (THREADS * 4); ++q) {
        uint32_t b[4];
        const int cnt = src.load_vals4((unsigned long long)u * kPruneUnit + (q * THREADS + t) * 4, n, b);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t key = b[e] & 0x7FFFFFFFu;
          nonfinite |= key >= kInfKey;  // (missing weights read as 0)
          const bool counts = e < cnt && (level == 0 || (key >> above) == prefix);
          const unsigned int who = __ballot_sync(FULL, counts);
          if (counts) {  // (lanes with equal digits add once: there may be a great many equal weights)
            const unsigned int digit = (key >> shift) & digit_mask, same = __match_any_sync(who, digit);
            if ((same & lt) == 0) atomicAdd(&sh.hist[digit], (unsigned int)__popc(same));
          }
        }
      }
    }, [&] { flush(ghist + level * kMaxBins); });
    if (nonfinite) set_status(&ctl->status, NSML_ERR_NONFINITE);
    if (!ok) return;
    find(ghist + level * kMaxBins, rem);
    prefix = prefix << digit_bits(level) | sh.out[0];
    rem = sh.out[1];
  }
  const uint32_t T = prefix;
  const unsigned int ties = sh.out[2], take = ties - rem + 1;  // ties to prune, lowest index first
  const bool ranked = take < ties;
  // a warp's 512 weights of a unit, 32 at a time: a ballot is a mask word
  auto fetch = [&](unsigned int u, uint32_t (&key)[16]) {
    const unsigned int i0 = u * kPruneUnit + warp * 512 + lane;
#pragma unroll
    for (int w = 0; w < 16; ++w) key[w] = i0 + w * 32 < n ? src.load1(i0 + w * 32) & 0x7FFFFFFFu : FULL;
  };
  if (ranked) {
    if (!run_phase(ctl, 6, units, sh, [&](unsigned int u) {
          uint32_t key[16];
          fetch(u, key);
          unsigned int c = 0;
#pragma unroll
          for (int w = 0; w < 16; ++w) c += key[w] == T;
          c = __reduce_add_sync(FULL, c);
          __syncthreads();
          if (lane == 0) sh.warp_ties[warp] = c;
          __syncthreads();
          if (t == 0) {
            unsigned int all = 0;
            for (int w = 0; w < NW; ++w) all += sh.warp_ties[w];
            unit_ties[u] = all;
          }
        }, [] {}))
      return;
    // exclusive prefix over the units, by one block
    if (!run_phase(ctl, 7, 1, sh, [&](unsigned int) {
          unsigned int carry = 0;
          for (unsigned int base = 0; base < units; base += THREADS) {
            const unsigned int c = base + t < units ? __ldcg(unit_ties + base + t) : 0u;
            unsigned int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const unsigned int up = __shfl_up_sync(FULL, incl, o);
              if (lane >= o) incl += up;
            }
            __syncthreads();
            if (lane == 31) sh.warp_ties[warp] = incl;
            __syncthreads();
            const unsigned int w = lane < NW ? sh.warp_ties[lane] : 0u;
            const unsigned int warps_before = __reduce_add_sync(FULL, lane < warp ? w : 0u), all = __reduce_add_sync(FULL, w);
            if (base + t < units) unit_ties[base + t] = carry + warps_before + incl - c;
            carry += all;
          }
        }, [] {}))
      return;
  }
  run_phase(ctl, 8, units, sh, [&](unsigned int u) {
    uint32_t key[16];
    fetch(u, key);
    unsigned int before = 0;  // ties before the warp's weights
    if (ranked) {
      unsigned int c = 0;
#pragma unroll
      for (int w = 0; w < 16; ++w) c += key[w] == T;
      c = __reduce_add_sync(FULL, c);
      __syncthreads();
      if (lane == 0) sh.warp_ties[warp] = c;
      __syncthreads();
      const unsigned int s = lane < warp ? sh.warp_ties[lane] : 0u;
      before = __ldcg(unit_ties + u) + __reduce_add_sync(FULL, s);
    }
#pragma unroll
    for (int w = 0; w < 16; ++w) {
      const bool tie = key[w] == T;
      const unsigned int bt = __ballot_sync(FULL, tie);
      const unsigned int word = __ballot_sync(FULL, key[w] < T || (tie && (!ranked || before + __popc(bt & lt) < take)));
      before += __popc(bt);
      const unsigned int first = u * kPruneUnit + warp * 512 + w * 32;
      if (lane == 0 && first < n) mask[first / 32] = word;
    }
  }, [] {});
}

}  // namespace nsml
