// Candidate list -> payload, in one kernel (Alg. 2 Step 3 read as: keep the k
// largest |g|, ties by lower index).
//
// The bucket pass leaves, per tile of the bucket, the candidates (every key >= lo)
// in index order with their number, and a histogram of the candidates inside the
// sampled window.  The threshold's bin is read off that histogram; it holds a few
// dozen keys, so one exchange between the blocks settles the rest:
//   0  every block scans the group counts (its share of the list: equal numbers of
//      candidates, so block order is index order and the work is balanced however
//      the candidates crowd) and finds the threshold's bin
//   1  copies its share into shared memory, counts the keys above the bin, appends
//      its keys inside the bin to the bin list                            | barrier
//   2  every block ranks the whole bin list (key descending, index ascending):
//      the threshold key T and the index of the last survivor with that key; the
//      position of its first survivor is the sum of the counts before it; writes
//      its survivors in order: index, and the value as float32 / fp16, or, for
//      int8, parked in raw_val
//   3  block 0 writes the header; int8 only, behind one more barrier: quantise
// A bin that holds more than kBinCap keys is refined by a histogram of its own (one
// more barrier each time) until it is short enough or a single key; then T is that
// key and the ties are ranked by the blocks' counts of them.  The same refinement
// finds the bin when the threshold lies above the window.
// If the list holds fewer than k candidates (fewer than k non-zero keys, or a
// misleading sample), the radix select over the bucket itself takes over
// (dense_select).
//
// What bounds the kernel is the number of dependent steps (a read from L2 0.7 us, a
// grid barrier 1.5-2 us), not its bytes; hence one exchange where a radix select on
// the list takes three, 1024 threads per block, and no separate kernel that makes
// the list contiguous.
#pragma once

#include "nsml_dense.cuh"

namespace nsml {

constexpr int kListThreads = 1024;
// Candidates a block keeps in shared memory (value and index); what does not fit is read again for the write phase.
constexpr int kListSmallCache = 8192, kListLargeCache = 22528;
constexpr size_t list_dyn_smem(int cache) { return (size_t)cache * 8; }
// The shortest lists run as ONE thread-block cluster of kListClusterBlocks blocks, whose barriers are the cluster's
// hardware barriers.
constexpr int kListClusterBlocks = 8;
constexpr double kListClusterMaxCandidates = 32768.0;  // expected candidates up to which the cluster shape is used

struct ListShared {
  FinalizeShared<kListThreads> f;
  unsigned int group_off[kMaxGroups + 1];   // list position of every group's first candidate
  unsigned int tile_off[kListThreads + 1];  // the same for the tiles of the window being copied
  unsigned long long warp_sum[kListThreads / 32];
  unsigned int total, window_total, before, first_idx, T, last_idx;
};

// The last i with off[i] <= pos (off ascending, off[0] <= pos, N a power of two).
template <int N>
__device__ __forceinline__ unsigned int last_at_most(const unsigned int* off, unsigned int pos) {
  unsigned int i = 0;
#pragma unroll
  for (int s = N / 2; s > 0; s >>= 1)
    if (off[i + s] <= pos) i += s;
  return i;
}

// VT: type of the listed values (bfloat16: packed entries).
template <int VT, int CACHE, bool CLUSTER>
__global__ void __launch_bounds__(kListThreads, 1) k_finalize(BucketSrc<VT> src, FinalizeParams p) {
  constexpr int THREADS = kListThreads, NW = THREADS / 32;
  constexpr unsigned int TILE = tile_elems<VT>();
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  constexpr unsigned int kMinShift = min_bin_shift<VT>();
  extern __shared__ __align__(16) uint32_t s_dyn[];
  uint32_t* c_val = s_dyn;
  uint32_t* c_idx = s_dyn + CACHE;
  __shared__ ListShared sh;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned int lt = (1u << lane) - 1u;
  const unsigned int G = gridDim.x, blk = blockIdx.x;
  const unsigned int k = (unsigned int)p.k;
  unsigned int barriers = 0;
  pdl_wait();

  // ---------------- phase 0: list positions of the groups; the threshold's bin ----------------
  const Window win = make_window<VT>(p.ctl);
  const unsigned int ngroups = (p.tiles + (1u << p.list.group_shift) - 1) >> p.list.group_shift;
  static_assert(kMaxGroups <= THREADS && kMaxBins == 4 * THREADS, "one group and four bins per thread");
  {
    const unsigned int mine = (unsigned int)t < ngroups ? __ldcg(p.list.group_count + t) : 0u;
    const uint4 b4 = __ldcg(reinterpret_cast<const uint4*>(p.list.window_hist) + t);
    const unsigned int bins[4] = {b4.x, b4.y, b4.z, b4.w};
    const unsigned int in_bins = b4.x + b4.y + b4.z + b4.w;
    unsigned int up_to = mine, from_here = in_bins;  // inclusive: groups up to this one, bins from this thread's on
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int a = __shfl_up_sync(FULL, up_to, o), b = __shfl_down_sync(FULL, from_here, o);
      if (lane >= o) up_to += a;
      if (lane + o < 32) from_here += b;
    }
    if (lane == 31) sh.f.scan[warp] = up_to;
    if (lane == 0) sh.f.tot[warp] = from_here;
    if (t == 0) sh.f.out[2] = 0;
    __syncthreads();
    unsigned int total = 0, window_total = 0, before = 0, above = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const unsigned int a = sh.f.scan[w], b = sh.f.tot[w];
      if (w < warp) before += a;
      if (w > warp) above += b;
      total += a;
      window_total += b;
    }
    sh.group_off[t] = before + up_to - mine;
    if (t == THREADS - 1) sh.group_off[kMaxGroups] = total;
    if (t == 0) { sh.total = total; sh.window_total = window_total; sh.before = 0; }
    // candidates above this thread's bins: those above the window and those in higher bins
    above += (total - window_total) + (from_here - in_bins);
    if (total >= k && above < k && k <= above + in_bins) {  // at most one thread
#pragma unroll
      for (int b = 3; b >= 0; --b) {
        if (k <= above + bins[b]) {
          sh.f.out[0] = t * 4 + b;
          sh.f.out[1] = k - above;
          sh.f.out[2] = bins[b];
          break;
        }
        above += bins[b];
      }
    }
    __syncthreads();
  }
  const unsigned int total = sh.total;
  if (total < k) {  // uniform over the grid
    dense_select<VT, THREADS, 8192, CLUSTER>(src, p, sh.f, s_dyn + 8192, s_dyn, 0);
    return;
  }
  const unsigned int share_lo = (unsigned int)((unsigned long long)blk * total / G);
  const unsigned int share_hi = (unsigned int)((unsigned long long)(blk + 1) * total / G);
  const bool resident = share_hi - share_lo <= (unsigned)CACHE;
  bool loaded = false;

  // Copies list positions [c0, c1) into shared memory.
  auto load_chunk = [&](unsigned int c0, unsigned int c1) {
    unsigned int pos = c0;
    while (pos < c1) {
      const unsigned int tile0 = last_at_most<kMaxGroups>(sh.group_off, pos) << p.list.group_shift;
      // a window of tiles from the group's first one on, a tile per thread
      const unsigned int cnt = tile0 + t < p.tiles ? __ldcg(p.list.tile_count + tile0 + t) : 0u;
      unsigned int in_window;
      const unsigned int excl = block_excl_scan(cnt, in_window, sh.f);
      const unsigned int start = sh.group_off[tile0 >> p.list.group_shift];
      sh.tile_off[t] = start + excl;
      if (t == 0) sh.tile_off[THREADS] = start + in_window;
      __syncthreads();
      const unsigned int end = min(c1, start + in_window);
      // A warp takes runs of 128 positions.  The tiles a run touches are usually few: the run's first tile is found with
      // two probes per lane, the others by comparing with the next tile boundaries, which the lanes hold.
      for (unsigned int run = pos + warp * 128; run < end; run += THREADS * 4) {
        const unsigned int run_end = min(end, run + 128);
        const unsigned int hi = 31 - __clz(__ballot_sync(FULL, sh.tile_off[lane * (THREADS / 32)] <= run));
        const unsigned int q0 = hi * 32 + 31 - __clz(__ballot_sync(FULL, sh.tile_off[hi * 32 + lane] <= run));
        const unsigned int bound = sh.tile_off[min(q0 + 1 + lane, (unsigned)THREADS)];  // where the next tiles start
        const unsigned int inside = __popc(__ballot_sync(FULL, bound < run_end));       // ... of which this many inside the run
        unsigned int v[4], i[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const unsigned int j = run + u * 32 + lane;
          unsigned int q = q0;
          if (inside == 32) {  // (more tiles than the lanes hold)
            q = last_at_most<THREADS>(sh.tile_off, min(j, end - 1));
          } else {
            for (unsigned int s = 0; s < inside; ++s) q += __shfl_sync(FULL, bound, s) <= j;
          }
          if (j < run_end) {
            i[u] = (tile0 + q) * TILE;
            const unsigned int at = i[u] + (j - sh.tile_off[q]);
            v[u] = __ldcg(p.list.val + at);
            if (VT == NSML_F32) i[u] += __ldcg(p.list.off + at);
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const unsigned int j = run + u * 32 + lane;
          if (j < run_end) {
            c_val[j - c0] = VT == NSML_F32 ? v[u] : v[u] << 16;
            c_idx[j - c0] = VT == NSML_F32 ? i[u] : i[u] + (v[u] >> 16);
          }
        }
      }
      pos = end;
      __syncthreads();
    }
  };
  // Calls f(number of entries in shared memory) for the block's share, a chunk at a time.
  auto for_chunks = [&](auto&& f) {
    for (unsigned int c0 = share_lo; c0 < share_hi; c0 += CACHE) {
      const unsigned int c1 = min(share_hi, c0 + CACHE);
      if (!resident || !loaded) load_chunk(c0, c1);
      loaded = true;
      f(c1 - c0);
      __syncthreads();  // the chunk has been used
    }
  };

  // ---------------- the threshold's bin: keys [bin_lo, bin_lo + 2^bin_shift), rem of bin_count kept ----------------
  unsigned int bin_lo, bin_shift, rem, bin_count;
  bool known = sh.f.out[2] != 0;
  if (known) {
    bin_lo = win.lo + (sh.f.out[0] << win.shift);
    bin_shift = win.shift;
    rem = sh.f.out[1];
    bin_count = sh.f.out[2];
  } else {  // the threshold lies above the window
    bin_lo = win.hi;
    bin_shift = 31;
    rem = k;
    bin_count = FULL;
  }
  for (int level = 0; !known || (bin_count > kBinCap && bin_shift > kMinShift); ++level) {  // at most three rounds: 31, 19, 7 bits
    const unsigned int shift = max(kMinShift, bin_shift > 12 ? bin_shift - 12 : 0u);
    const unsigned int span = 1u << bin_shift;
    __syncthreads();  // sh.f.out has been read
    for (int b = t; b < kMaxBins; b += THREADS) sh.f.hist[b] = 0;
    __syncthreads();
    for_chunks([&](unsigned int cnt) {
      for (unsigned int j = t; j < cnt; j += THREADS) {
        const unsigned int rel = (c_val[j] & 0x7FFFFFFFu) - bin_lo;
        if (rel < span) atomicAdd(&sh.f.hist[rel >> shift], 1u);
      }
    });
    flush_hist<kMaxBins>(sh.f, p.hist + level * kMaxBins);
    if (!grid_barrier<CLUSTER>(p.ctl, ++barriers * G, sh.f)) return;
    resolve_digit<kMaxBins>(p.hist + level * kMaxBins, rem, sh.f);
    bin_lo += sh.f.out[0] << shift;
    bin_shift = shift;
    rem = sh.f.out[1];
    bin_count = sh.f.out[2];
    known = true;
  }
  const bool listed = bin_count <= kBinCap;  // else the bin is a single key
  const unsigned int bin_span = 1u << bin_shift;

  // ---------------- phase 1: count the keys above the bin and inside it ----------------
  {
    unsigned int above = 0, inside = 0;
    bool first = true;
    for_chunks([&](unsigned int cnt) {
      if (first && t == 0) sh.first_idx = c_idx[0];
      first = false;
      for (unsigned int j = t; j < cnt; j += THREADS) {
        const unsigned int key = c_val[j] & 0x7FFFFFFFu;
        if (key < bin_lo) continue;
        if (key - bin_lo >= bin_span) {
          ++above;
        } else {
          ++inside;
          if (listed) {
            const unsigned int slot = atomicAdd(&p.ctl->listed, 1u);
            if (slot < kBinCap) p.bin_list[slot] = make_uint2(key, c_idx[j]);
          }
        }
      }
    });
    const unsigned long long both = block_sum(((unsigned long long)above << 32) | inside, sh.f);
    if (t == 0) p.block_counts[blk] = both;
  }
  if (!grid_barrier<CLUSTER>(p.ctl, ++barriers * G, sh.f)) return;

  // ---------------- phase 2: the exact threshold; write the survivors in index order ----------------
  uint2* s_bin = reinterpret_cast<uint2*>(sh.f.hist);
  static_assert(sizeof(uint2) * kBinCap <= sizeof(sh.f.hist), "the bin list fits the histogram");
  unsigned long long before, all;
  {
    if (listed)
      for (unsigned int i = t; i < bin_count; i += THREADS) s_bin[i] = __ldcg(p.bin_list + i);
    before = all = 0;  // every warp adds up the counts for itself: no block barriers
    for (unsigned int b = lane; b < G; b += 32) {
      const unsigned long long w = __ldcg(p.block_counts + b);
      all += w;
      if (b < blk) before += w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      all += __shfl_xor_sync(FULL, all, o);
      before += __shfl_xor_sync(FULL, before, o);
    }
    __syncthreads();  // s_bin is complete
  }
  if ((unsigned int)(all >> 32) + rem != k || (unsigned int)all != bin_count) {
    if (t == 0) set_status(&p.ctl->status, NSML_ERR_INTERNAL);
    return;
  }
  uint32_t T = (bin_lo + ((1u << kMinShift) - 1u)) & ~((1u << kMinShift) - 1u);  // the bin's key, where it holds one
  uint32_t last_idx = 0;
  unsigned int pos = (unsigned int)(before >> 32);  // payload position of the block's first survivor
  unsigned int quota = 0;                            // single-key bin: ties the block keeps, lowest index first
  if (listed) {
    for (unsigned int i = t; i < bin_count; i += THREADS) {
      const uint2 me = s_bin[i];
      unsigned int rank = 0;
      for (unsigned int q = 0; q < bin_count; ++q) {
        const uint2 o = s_bin[q];
        rank += o.x > me.x || (o.x == me.x && o.y < me.y);
      }
      if (rank == rem - 1) {  // exactly one entry: the last survivor
        sh.T = me.x;
        sh.last_idx = me.y;
      }
      if (rank < rem && me.y < sh.first_idx && share_hi > share_lo) atomicAdd(&sh.before, 1u);
    }
    __syncthreads();
    T = sh.T;
    last_idx = sh.last_idx;
    pos += sh.before;
  } else {
    const unsigned int ties_before = (unsigned int)before;
    quota = rem > ties_before ? rem - ties_before : 0u;
    pos += min(ties_before, rem);
  }
  uint32_t* out_idx = reinterpret_cast<uint32_t*>(p.payload + p.P.idx_off);
  for_chunks([&](unsigned int cnt) {
    // a warp owns a contiguous run of the chunk: it counts its survivors, then writes them behind the warps before it
    const unsigned int per = ((cnt + NW - 1) / NW + 31) / 32 * 32;
    const unsigned int run_lo = min(cnt, warp * per), run_hi = min(cnt, run_lo + per);
    unsigned int n_sure = 0, n_tied = 0;
    for (unsigned int j = run_lo + lane; j < run_hi; j += 32) {
      const uint32_t key = c_val[j] & 0x7FFFFFFFu;
      const bool tied = key == T;
      n_sure += key > T || (listed && tied && c_idx[j] <= last_idx);
      n_tied += !listed && tied;
    }
    n_sure = __reduce_add_sync(FULL, n_sure);
    n_tied = __reduce_add_sync(FULL, n_tied);
    if (lane == 0) sh.warp_sum[warp] = ((unsigned long long)n_sure << 32) | n_tied;
    __syncthreads();
    unsigned long long up_to = sh.warp_sum[lane];  // NW == 32: a warp sum per lane
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long a = __shfl_up_sync(FULL, up_to, o);
      if (lane >= o) up_to += a;
    }
    const unsigned long long chunk_all = __shfl_sync(FULL, up_to, 31);
    const unsigned long long warps_before = warp == 0 ? 0ull : __shfl_sync(FULL, up_to, (warp + 31) & 31);
    unsigned int sure = (unsigned int)(warps_before >> 32), tied = (unsigned int)warps_before;
    for (unsigned int j0 = run_lo; j0 < run_hi; j0 += 32) {
      const unsigned int j = j0 + lane;
      const bool live = j < run_hi;
      const uint32_t bits = live ? c_val[j] : 0u, idx = live ? c_idx[j] : 0u;
      const uint32_t key = bits & 0x7FFFFFFFu;
      const bool is_tied = live && !listed && key == T;
      const bool is_sure = live && (key > T || (listed && key == T && idx <= last_idx));
      const unsigned int bs = __ballot_sync(FULL, is_sure), bt = __ballot_sync(FULL, is_tied);
      const unsigned int s_mine = sure + __popc(bs & lt), t_mine = tied + __popc(bt & lt);
      if (is_sure || (is_tied && t_mine < quota)) {
        const unsigned int at = pos + s_mine + min(t_mine, quota);
        out_idx[at] = idx;
        put_value(p, at, bits);
      }
      sure += __popc(bs);
      tied += __popc(bt);
    }
    const unsigned int c_sure = (unsigned int)(chunk_all >> 32), c_tied = (unsigned int)chunk_all;
    pos += c_sure + min(c_tied, quota);
    quota -= min(c_tied, quota);
  });

  // ---------------- phase 3: the header; int8: quantise ----------------
  if (blk == 0 && t == 0) write_header(p);
  if (p.bits != NSML_BITS_INT8) return;  // float32 and fp16 values are in the payload already
  if (!grid_barrier<CLUSTER>(p.ctl, ++barriers * G, sh.f)) return;
  quantize_all(p, sh.f);
}

}  // namespace nsml
