// Small bucket -> payload in one kernel: one block, or one thread-block cluster of
// kSmallBlocks blocks that hold the whole bucket in shared memory.
//
// A bucket of some ten thousand elements is launches and latency: two or three kernels
// and four or five grid barriers through global memory take 25 us for what is read in
// one.  Here the bucket is read once (with the residual added where there is one), the
// radix select (12 + 12 + 7 bits of the magnitude key; Alg. 2 Step 3 read as: keep the k
// largest |g|, ties by lower index) runs on the shared-memory copy, its histograms are
// summed through distributed shared memory, and the barriers are the cluster's.
//
// Measured (one B200, whole call, int8, kept fraction 0.001 / 0.1 / 0.5): 12,289 elements 25 / 27 / 27 us with the other
// strategies, 12-13 us here; 65,536 elements 19 / 26 / 29 -> 13.5 / 16 / 18;
// 131,072 elements 19 / 28 / 29 -> 17 / 19 / 24; at 200,000 elements it is even, hence the limit.  One block instead of
// the cluster pays up to about 8,000 elements.  The keys of the first digit's bin by themselves where they are few, instead
// of two more digits: 8,192 elements at 0.1 11.0 -> 10.0, 12,289 12.1 -> 10.9, 40,000 14.6 -> 13.1, 163,840 at 0.001 19.1 -> 16.9.
#pragma once

#include <cooperative_groups.h>

#include "nsml_list.cuh"

namespace nsml {

constexpr int kSmallThreads = 1024;
constexpr int kSmallBlocks = 8;
constexpr unsigned int kSmallOneBlock = 8192;      // largest bucket that one block takes on its own
constexpr unsigned int kSmallPerBlock = 20480;     // elements a block holds at most
constexpr int64_t kSmallMaxN = (int64_t)kSmallBlocks * kSmallPerBlock;
constexpr unsigned int kSmallKeys = kSmallThreads;  // keys of the first digit's bin that are looked at one per thread

struct SmallShared {
  unsigned int hist[kMaxBins];
  unsigned int tot[kSmallThreads / 32], out[3], slice[kSmallBlocks], listed;
  uint2 warp_sum[kSmallThreads / 32], block_sum[kSmallBlocks];
  float qmax[kSmallThreads / 32];
};

// per_block: elements of a block, a multiple of 128.  BLOCKS: 1 or kSmallBlocks.
template <int DTYPE, int BLOCKS>
__global__ void __launch_bounds__(kSmallThreads, 1)
k_select_small(BucketSrc<DTYPE> src, FinalizeParams p, unsigned int per_block, int keep_status) {
  namespace cg = cooperative_groups;
  constexpr int THREADS = kSmallThreads, NW = THREADS / 32;
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  extern __shared__ __align__(16) uint32_t s_val[];  // the block's elements, as float32 bit patterns
  __shared__ SmallShared sh;
  cg::cluster_group cluster = cg::this_cluster();
  const unsigned int rank = BLOCKS == 1 ? 0u : cluster.block_rank();
  auto sync_all = [&] { if (BLOCKS == 1) __syncthreads(); else cluster.sync(); };
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned int n = (unsigned int)p.n, k = (unsigned int)p.k;
  const unsigned int lo = min(n, rank * per_block), E = min(n, lo + per_block) - lo;
  for (int b = t; b < kMaxBins; b += THREADS) sh.hist[b] = 0;
  __syncthreads();
  pdl_wait();
  pdl_launch_dependents();
  if (rank == 0 && t == 0 && !keep_status) p.ctl->status = NSML_OK;
  if (t == 0) sh.listed = 0;

  // ---------------- load; histogram of digit 0 ----------------
  bool nonfinite = false;
  unsigned int zeros = 0;  // zero keys would all hit bin 0
  for (unsigned int i = t * 4; i < E; i += THREADS * 4) {
    uint32_t b[4];
    const unsigned int at = lo + i;
    int cnt;
    if (p.residual == nullptr) {
      cnt = src.load_vals4(at, n, b);
    } else {
      const BucketSrc<DTYPE> bare{src.grad, nullptr};
      cnt = bare.load_vals4(at, n, b);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (e < cnt) {
          const float sum = __fadd_rn(__uint_as_float(b[e]), p.residual[at + e]);
          p.residual[at + e] = sum;
          b[e] = src.pruned(at + e) ? 0u : __float_as_uint(sum);
        }
      }
    }
    *reinterpret_cast<uint4*>(s_val + i) = make_uint4(b[0], b[1], b[2], b[3]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t key = b[e] & 0x7FFFFFFFu;
      nonfinite |= key >= kInfKey;  // missing entries read as 0
      if (e < cnt) {
        if (key == 0) ++zeros; else atomicAdd(&sh.hist[key >> digit_shift(0)], 1u);
      }
    }
  }
  zeros = __reduce_add_sync(FULL, zeros);
  if (lane == 0 && zeros) atomicAdd(&sh.hist[0], zeros);

  // ---------------- the threshold, digit by digit ----------------
  unsigned int prefix = 0, rem = k;
#pragma unroll
  for (int level = 0; level < 3; ++level) {
    const int bins = 1 << digit_bits(level);
    if (BLOCKS == 1) {
      __syncthreads();
      unsigned int own[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) own[b] = t * 4 + b < bins ? sh.hist[t * 4 + b] : 0u;
      find_digit_from_top<4, THREADS>(own, rem, sh.tot, sh.out);
    } else {
      cluster.sync();  // the counts of every block are complete
      // this block's slice of the bins, summed over the blocks
      const int slice = bins / kSmallBlocks;
      unsigned int own = 0;
      if (t < slice) {
#pragma unroll
        for (int b = 0; b < kSmallBlocks; ++b) own += cluster.map_shared_rank(sh.hist, b)[rank * slice + t];
      }
      unsigned int incl = own;  // this bin and those of the higher lanes
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned int down = __shfl_down_sync(FULL, incl, o);
        if (lane + o < 32) incl += down;
      }
      if (lane == 0) sh.tot[warp] = incl;
      __syncthreads();
      const unsigned int w = sh.tot[lane];
      const unsigned int higher = __reduce_add_sync(FULL, lane > warp ? w : 0u), all = __reduce_add_sync(FULL, w);
      if (t < kSmallBlocks) *cluster.map_shared_rank(&sh.slice[rank], t) = all;
      cluster.sync();  // the slices' totals are in place; nobody reads the counts any more
      const unsigned int s = lane < kSmallBlocks ? sh.slice[lane] : 0u;
      const unsigned int above = __reduce_add_sync(FULL, lane > (int)rank ? s : 0u) + higher + incl - own;
      if (above < rem && rem <= above + own) {  // one thread of the cluster
        for (int b = 0; b < kSmallBlocks; ++b) {
          unsigned int* out = cluster.map_shared_rank(sh.out, b);
          out[0] = rank * slice + t;
          out[1] = rem - above;
          out[2] = own;
        }
      }
      if (level < 2)
        for (int b = t; b < kMaxBins; b += THREADS) sh.hist[b] = 0;
      cluster.sync();
    }
    prefix = (prefix << digit_bits(level)) | sh.out[0];
    rem = sh.out[1];
    if (level == 2) break;
    if (level == 0 && sh.out[2] <= kSmallKeys) {
      // The bin's keys, each block's in its histogram's place, then one per thread of every block: the threshold bit by
      // bit.  (Two more digits take six barriers of the cluster and two passes over the elements.  Up to four keys per
      // thread: 4 us slower than one, whatever the bin holds.)
      const unsigned int in_bin = sh.out[2];
      if (BLOCKS == 1) __syncthreads();
      for (unsigned int i = t * 4; i < E; i += THREADS * 4) {
        const uint4 q = *reinterpret_cast<const uint4*>(s_val + i);
        const uint32_t b[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t key = b[e] & 0x7FFFFFFFu;
          if (i + e < E && (key >> digit_shift(0)) == prefix) sh.hist[atomicAdd(&sh.listed, 1u)] = key;
        }
      }
      sync_all();
      uint32_t key = 0;
      if (BLOCKS == 1) {
        if ((unsigned)t < in_bin) key = sh.hist[t];
      } else {
        const unsigned int count = lane < BLOCKS ? *cluster.map_shared_rank(&sh.listed, lane) : 0u;
        unsigned int at = t, from = 0;
#pragma unroll
        for (int b = 0; b < BLOCKS; ++b) {
          const unsigned int c = __shfl_sync(FULL, count, b);
          if (from == (unsigned)b && at >= c) {
            at -= c;
            ++from;
          }
        }
        if ((unsigned)t < in_bin) key = cluster.map_shared_rank(sh.hist, from)[at];
      }
      prefix <<= digit_shift(0);
      for (uint32_t bit = 1u << (digit_shift(0) - 1); bit != 0; bit >>= 1)
        if ((unsigned)__syncthreads_count((unsigned)t < in_bin && key >= (prefix | bit)) >= rem) prefix |= bit;
      rem -= __syncthreads_count((unsigned)t < in_bin && key > prefix);
      break;
    }
    if (BLOCKS == 1) {
      for (int b = t; b < kMaxBins; b += THREADS) sh.hist[b] = 0;
      __syncthreads();
    }
    const int shift = digit_shift(level), next = digit_shift(level + 1);
    const unsigned int mask = (1u << digit_bits(level + 1)) - 1u;
    zeros = 0;
    for (unsigned int i = t * 4; i < E; i += THREADS * 4) {
      const uint4 q = *reinterpret_cast<const uint4*>(s_val + i);
      const uint32_t b[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const uint32_t key = b[e] & 0x7FFFFFFFu;
        if (i + e < E && (key >> shift) == prefix) {
          if (key == 0) ++zeros; else atomicAdd(&sh.hist[(key >> next) & mask], 1u);
        }
      }
    }
    if (prefix == 0) {
      zeros = __reduce_add_sync(FULL, zeros);
      if (lane == 0 && zeros) atomicAdd(&sh.hist[0], zeros);
    }
  }
  const uint32_t T = prefix;
  const unsigned int r = rem;  // ties (key == T) to keep, lowest index first
  if (nonfinite) set_status(&p.ctl->status, NSML_ERR_NONFINITE);

  // ---------------- count: a warp takes a contiguous run, four elements per lane ----------------
  const unsigned int per_warp = ((E + NW - 1) / NW + 127) / 128 * 128;
  const unsigned int run_lo = min(E, warp * per_warp), run_hi = min(E, run_lo + per_warp);
  unsigned int n_sure = 0, n_tied = 0;
  for (unsigned int i = run_lo + lane * 4; i < run_hi; i += 128) {
    const uint4 q = *reinterpret_cast<const uint4*>(s_val + i);
    const uint32_t b[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t key = b[e] & 0x7FFFFFFFu;
      n_sure += i + e < run_hi && key > T;
      n_tied += i + e < run_hi && key == T;
    }
  }
  n_sure = __reduce_add_sync(FULL, n_sure);
  n_tied = __reduce_add_sync(FULL, n_tied);
  if (lane == 0) sh.warp_sum[warp] = make_uint2(n_sure, n_tied);
  __syncthreads();
  const uint2 ws = sh.warp_sum[lane];
  unsigned int sure = __reduce_add_sync(FULL, lane < warp ? ws.x : 0u), tied = __reduce_add_sync(FULL, lane < warp ? ws.y : 0u);
  if (BLOCKS > 1) {
    const uint2 all = make_uint2(__reduce_add_sync(FULL, ws.x), __reduce_add_sync(FULL, ws.y));
    if (t < kSmallBlocks) *cluster.map_shared_rank(&sh.block_sum[rank], t) = all;
    cluster.sync();
    const uint2 bs = lane < (int)rank ? sh.block_sum[lane] : make_uint2(0u, 0u);
    sure += __reduce_add_sync(FULL, bs.x);
    tied += __reduce_add_sync(FULL, bs.y);
  }

  // ---------------- write the survivors in index order ----------------
  uint32_t* out_idx = reinterpret_cast<uint32_t*>(p.payload + p.P.idx_off);
  for (unsigned int i0 = run_lo; i0 < run_hi; i0 += 128) {
    const unsigned int i = i0 + lane * 4;
    uint4 q = make_uint4(0u, 0u, 0u, 0u);
    if (i < run_hi) q = *reinterpret_cast<const uint4*>(s_val + i);
    const uint32_t b[4] = {q.x, q.y, q.z, q.w};
    unsigned int fs = 0, ft = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const uint32_t key = b[e] & 0x7FFFFFFFu;
      fs |= (unsigned int)(i + e < run_hi && key > T) << e;
      ft |= (unsigned int)(i + e < run_hi && key == T) << e;
    }
    if (__ballot_sync(FULL, (fs | ft) != 0) == 0) continue;
    const unsigned int mine = __popc(fs) | (__popc(ft) << 16);  // at most 128 each in a warp
    unsigned int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int up = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += up;
    }
    unsigned int s_mine = sure + ((incl - mine) & 0xFFFFu), t_mine = tied + ((incl - mine) >> 16);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const bool is_sure = fs & (1u << e), is_tied = ft & (1u << e);
      if (is_sure || (is_tied && t_mine < r)) {
        const unsigned int at = s_mine + min(t_mine, r), idx = lo + i + e;
        if (at < k) {
          out_idx[at] = idx;
          put_value(p, at, b[e]);
          if (p.residual != nullptr && p.bits != NSML_BITS_INT8 && b[e] != 0) p.residual[idx] = not_carried(p, b[e]);
        }
      }
      s_mine += is_sure;
      t_mine += is_tied;
    }
    const unsigned int total = __shfl_sync(FULL, incl, 31);
    sure += total & 0xFFFFu;
    tied += total >> 16;
  }
  if (rank == 0 && t == 0) write_header(p);
  if (p.bits != NSML_BITS_INT8) return;  // (nobody reads this block's shared memory any more)

  // ---------------- int8: quantise ----------------
  __threadfence();
  sync_all();
  const unsigned int blocks = (k + NSML_QBLOCK - 1) / NSML_QBLOCK;
  for (unsigned int q0 = rank * (NW / 4); q0 < blocks; q0 += BLOCKS * (NW / 4)) {
    const unsigned int q = q0 + (warp >> 2);
    quantize_group(p, p.residual, sh.qmax, q, q < blocks, q < blocks ? min(k, (q + 1) * NSML_QBLOCK) - q * NSML_QBLOCK : 0u,
                   [&](unsigned int j) { return __ldcg(p.raw_val + (size_t)q * NSML_QBLOCK + j); },
                   [&](unsigned int j) { return __ldcg(out_idx + (size_t)q * NSML_QBLOCK + j); });
  }
}

}  // namespace nsml
