// Candidate list -> payload (Alg. 2 Step 3 read as: keep the k largest |g|, ties by
// lower index).
//
// The bucket pass leaves, per tile of the bucket, the candidates (every key >= lo) in
// index order with their number; a histogram of the candidates inside the sampled
// window; and those candidates once more, by bin.  k_emit turns that into the payload
// with no barrier between blocks:
//   every block scans the counts (list positions of the tiles, total) and finds the
//   threshold's bin; the bin's few dozen keys, ranked (key descending, index
//   ascending), give the threshold key T and the index of the last survivor with that
//   key.  A bin that holds one key (bfloat16) needs no list: T is that key, and ties
//   are kept by their rank.
//   The list is then taken in chunks of 2048 candidates, which blocks draw by ticket: a
//   block loads a chunk into registers, counts its survivors, publishes the count,
//   adds up the counts of the chunks before it (which have been drawn earlier, so the
//   blocks that hold them are running: the wait cannot deadlock), and writes the
//   survivors in order: index and value; int8: payload blocks of 1024 values that lie
//   inside the chunk are quantised from shared memory, one that it shares with other
//   chunks by whichever of them delivers the last value.
//
// What bounds the kernel is the number of dependent steps (a read from L2 0.7 us), not
// its bytes.  As a cooperative kernel whose blocks kept the chunk in shared memory and
// exchanged the bin's keys at a grid barrier it took 20 us for 330k candidates, plus 2
// us until a cooperative grid starts behind the bucket pass.
//
// Calls that this does not cover (fewer than k candidates because of a misleading sample; a threshold above the window;
// a bin of many keys that turn out not to be one key) take more rounds (general_select).
#pragma once

#include "nsml_finalize.cuh"

namespace nsml {

// The last i with off[i] <= pos (off ascending, off[0] <= pos, N a power of two).
template <int N>
__device__ __forceinline__ unsigned int last_at_most(const unsigned int* off, unsigned int pos) {
  unsigned int i = 0;
#pragma unroll
  for (int s = N / 2; s > 0; s >>= 1)
    if (off[i + s] <= pos) i += s;
  return i;
}

// The same by a warp for one position, over kMaxGroups entries.
__device__ __forceinline__ unsigned int warp_last_at_most(const unsigned int* off, unsigned int pos) {
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  static_assert(kMaxGroups == 32 * 32 * 8, "three levels of probes");
  const unsigned int lane = threadIdx.x & 31;
  const unsigned int a = 31 - __clz(__ballot_sync(FULL, off[lane * 256] <= pos));
  const unsigned int b = a * 32 + 31 - __clz(__ballot_sync(FULL, off[a * 256 + lane * 8] <= pos));
  return b * 8 + 31 - __clz(__ballot_sync(FULL, lane < 8 && off[b * 8 + lane] <= pos));
}

// Loads list positions run .. run_end - 1 (at most 32 * U) into the registers of a warp: v[u], i[u] = value and index
// of position run + u * 32 + lane.  off: list positions of the groups.
template <int VT, int U>
__device__ __forceinline__ void fetch_run(const TileList& list, const unsigned int* off, unsigned int tiles, unsigned int run,
                                          unsigned int run_end, uint32_t (&v)[U], uint32_t (&i)[U]) {
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  constexpr unsigned int TILE = tile_elems<VT>();
  const unsigned int lane = threadIdx.x & 31;
  auto load = [&](int u, unsigned int tile, unsigned int within) {
    const unsigned int at = tile * TILE + within;
    v[u] = __ldcg(list.val + at);
    i[u] = tile * TILE;
    if (VT == NSML_F32) i[u] += __ldcg(list.off + at);
  };
#pragma unroll
  for (int u = 0; u < U; ++u) v[u] = i[u] = 0;
  if (list.group_shift == 0) {
    // A group is a tile.  The tiles a run touches are usually few: the first is found by probing, the others by
    // comparing with the next tile boundaries, which the lanes hold.
    const unsigned int q0 = warp_last_at_most(off, run);
    const unsigned int bound = off[min(q0 + 1 + lane, (unsigned)kMaxGroups)];            // where the next tiles start
    const unsigned int inside = __popc(__ballot_sync(FULL, bound < run_end));  // ... of which this many inside the run
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned int j = run + u * 32 + lane;
      unsigned int q = q0;
      if (inside == 32) {  // (more tiles than the lanes hold)
        q = last_at_most<kMaxGroups>(off, min(j, run_end - 1));
      } else {
        for (unsigned int s = 0; s < inside; ++s) q += __shfl_sync(FULL, bound, s) <= j;
      }
      if (j < run_end) load(u, q, j - off[q]);
    }
  } else {
    // Buckets of more than kMaxGroups tiles: the counts of 64 tiles from the first one's group on are read and summed up,
    // two per lane; a lane finds its tiles by a search over the lanes.  Usually one round does.
    for (unsigned int pos = run; pos < run_end;) {
      const unsigned int g = warp_last_at_most(off, pos), tile0 = (g << list.group_shift) + lane * 2;
      const unsigned int c0 = tile0 < tiles ? __ldcg(list.tile_count + tile0) : 0u;
      const unsigned int c1 = tile0 + 1 < tiles ? __ldcg(list.tile_count + tile0 + 1) : 0u;
      unsigned int incl = c0 + c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned int up = __shfl_up_sync(FULL, incl, o);
        if (lane >= (unsigned)o) incl += up;
      }
      const unsigned int s0 = off[g] + incl - c0 - c1, s1 = s0 + c0;  // where the lane's two tiles start
      const unsigned int end = min(run_end, off[g] + __shfl_sync(FULL, incl, 31));
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const unsigned int j = run + u * 32 + lane;
        unsigned int a = 0;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1)
          if (__shfl_sync(FULL, s0, a + s) <= j) a += s;
        const unsigned int first = __shfl_sync(FULL, s0, a), second = __shfl_sync(FULL, s1, a);
        if (j >= pos && j < end) load(u, (g << list.group_shift) + a * 2 + (j >= second), j - (j >= second ? second : first));
      }
      pos = end;
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (VT != NSML_F32) {  // packed: offset << 16 | bfloat16 bits
      i[u] += v[u] >> 16;
      v[u] <<= 16;
    }
  }
}

// What every block of the list stage works out first: the list positions of the groups, the number of candidates, and
// the bin of the window that holds the k-th largest key.
template <int THREADS>
struct ListScan {
  __align__(16) unsigned int off[kMaxGroups + 4];  // list position of every group's first candidate; the total behind the last
  unsigned int groups[THREADS / 32], bins[THREADS / 32];
  unsigned int total, in_window;
  unsigned int bin, rem, bin_count;  // bin_count = 0: the threshold lies above the window, or there are fewer than k candidates
};

template <int THREADS>
__device__ __forceinline__ void scan_list(const FinalizeParams& p, unsigned int k, ListScan<THREADS>& sc) {
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  constexpr int NW = THREADS / 32, ROWS = kMaxGroups / (NW * 128), QUADS = kMaxBins / (THREADS * 4);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned int ngroups = (p.tiles + (1u << p.list.group_shift) - 1) >> p.list.group_shift;
  // a warp takes ROWS rows of 128 consecutive counts, four per lane; a thread takes QUADS * 4 consecutive bins
  uint4 g[ROWS], b[QUADS];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const unsigned int at = (warp * ROWS + r) * 128 + lane * 4;
    g[r] = at < ngroups ? __ldcg(reinterpret_cast<const uint4*>(p.list.group_count + at)) : make_uint4(0u, 0u, 0u, 0u);
  }
#pragma unroll
  for (int q = 0; q < QUADS; ++q) b[q] = __ldcg(reinterpret_cast<const uint4*>(p.list.window_hist) + t * QUADS + q);
  unsigned int excl[ROWS], warp_groups = 0;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    excl[r] = warp_groups;
    if ((warp * ROWS + r) * 128 >= ngroups) continue;  // (nothing there)
    const unsigned int mine = g[r].x + g[r].y + g[r].z + g[r].w;
    unsigned int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int up = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += up;
    }
    excl[r] = warp_groups + incl - mine;
    warp_groups += __shfl_sync(FULL, incl, 31);
  }
  unsigned int my_bins = 0;
#pragma unroll
  for (int q = 0; q < QUADS; ++q) my_bins += b[q].x + b[q].y + b[q].z + b[q].w;
  unsigned int from_here = my_bins;  // this thread's bins and those of the higher lanes
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int down = __shfl_down_sync(FULL, from_here, o);
    if (lane + o < 32) from_here += down;
  }
  if (lane == 0) {
    sc.groups[warp] = warp_groups;
    sc.bins[warp] = from_here;
  }
  if (t == 0) sc.bin_count = 0;
  __syncthreads();
  const unsigned int wg = lane < NW ? sc.groups[lane] : 0u, wb = lane < NW ? sc.bins[lane] : 0u;
  const unsigned int before = __reduce_add_sync(FULL, lane < warp ? wg : 0u), total = __reduce_add_sync(FULL, wg);
  unsigned int above = __reduce_add_sync(FULL, lane > warp ? wb : 0u);
  const unsigned int in_window = __reduce_add_sync(FULL, wb);
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const unsigned int at = before + excl[r];
    *reinterpret_cast<uint4*>(sc.off + (warp * ROWS + r) * 128 + lane * 4) =
        make_uint4(at, at + g[r].x, at + g[r].x + g[r].y, at + g[r].x + g[r].y + g[r].z);
  }
  if (t == 0) {
    sc.off[kMaxGroups] = sc.total = total;
    sc.in_window = in_window;
  }
  // candidates above this thread's bins: those above the window and those in higher bins
  above += (total - in_window) + (from_here - my_bins);
  if (total >= k && above < k && k <= above + my_bins) {  // at most one thread
#pragma unroll
    for (int q = QUADS - 1; q >= 0; --q) {
      const unsigned int c[4] = {b[q].x, b[q].y, b[q].z, b[q].w};
#pragma unroll
      for (int e = 3; e >= 0; --e) {
        if (above < k && k <= above + c[e]) {
          sc.bin = (t * QUADS + q) * 4 + e;
          sc.rem = k - above;
          sc.bin_count = c[e];
        }
        above += c[e];
      }
    }
  }
  __syncthreads();
}

// ------------------------------------------------------------------------
// k_emit
// ------------------------------------------------------------------------
constexpr int kEmitThreads = 512;
constexpr int kEmitPer = kChunk / kEmitThreads;  // candidates per thread of the (smaller) chunk
constexpr int kLargeChunk = 2 * kChunk;
constexpr unsigned int kMaxBinRoom = 2048;

struct EmitShared {
  ListScan<kEmitThreads> sc;
  uint2 warp_sum[kEmitThreads / 32], back_sum[kEmitThreads / 32];  // (above the threshold, tied with it)
  float qmax[kEmitThreads / 32];
  unsigned int ticket[2], T, last_idx, done[2];
  union {
    uint2 bin[kMaxBinRoom];  // the threshold's bin: (key, index)
    struct {
      uint32_t val[kLargeChunk], idx[kLargeChunk];  // int8: the chunk's survivors
    } kept;
    struct {
      unsigned int hist[kMaxBins], tot[kEmitThreads / 32], out[3];
    } general;
  };
};

// Polls a published sum (bit 63 set) with a bounded number of attempts; 0 = gave up.
__device__ __forceinline__ unsigned long long wait_sum(const unsigned long long* at) {
  unsigned long long v;
  for (int polls = 0; polls < kMaxPolls; ++polls) {
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(at) : "memory");
    if (v >> 63) return v;
    if (polls > 64) __nanosleep(32);
  }
  return 0;
}
__device__ __forceinline__ void publish_sum(unsigned long long* at, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(at), "l"(v | (1ull << 63)) : "memory");
}
// sums: keys above the threshold in bits 31.., keys equal to it (where those are kept by rank) in bits 0..30
__device__ __forceinline__ unsigned int sure_of(unsigned long long s) { return (unsigned int)(s >> 31) & 0x7FFFFFFFu; }
__device__ __forceinline__ unsigned int tied_of(unsigned long long s) { return (unsigned int)s & 0x7FFFFFFFu; }

// 128 threads (four warps) turn values get(j), j < cnt <= 1024, into the codes and the scale of payload block qb; with a
// residual, what the codes do not carry stays at the values' indices index(j) (a zero leaves its place alone: it may be a
// pruned parameter's, whose sum stays; and code 0 is +0.0, which taken out of -0.0 leaves -0.0).
// Called by every thread of the block (it holds block barriers); live: the group has a block.
template <class Get, class Index>
__device__ __forceinline__ void quantize_group(const FinalizeParams& p, float* residual, float* s_qmax, unsigned int qb, bool live, unsigned int cnt,
                                               Get&& get, Index&& index) {
  const int gt = threadIdx.x & 127, warp = threadIdx.x >> 5;
  float v[8], m = 0.f;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const unsigned int j = e * 128 + gt;
    v[e] = live && j < cnt ? get(j) : 0.f;
    m = fmaxf(m, fabsf(v[e]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  __syncthreads();  // s_qmax of the previous round has been read
  if ((threadIdx.x & 31) == 0) s_qmax[warp] = m;
  __syncthreads();
  if (!live) return;
  const float* q = s_qmax + (warp & ~3);
  m = fmaxf(fmaxf(q[0], q[1]), fmaxf(q[2], q[3]));
  const float scale = __fdiv_rn(m, 127.0f), inv = __fdiv_rn(1.0f, scale);
  if (gt == 0) reinterpret_cast<float*>(p.payload + p.P.scale_off)[qb] = scale;
  signed char* out = reinterpret_cast<signed char*>(p.payload + p.P.val_off) + (size_t)qb * NSML_QBLOCK;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const unsigned int j = e * 128 + gt;
    if (j < cnt) {
      const int code = encode_i8(v[e], scale, inv);
      out[j] = (signed char)code;
      if (residual != nullptr && v[e] != 0.0f) residual[index(j)] = __fsub_rn(v[e], decode_i8(code, scale));
    }
  }
}

// What the survivors are.
struct Choice {
  uint32_t T;             // the threshold key
  unsigned int last_idx;  // not ranked: keys equal to T survive up to this index ...
  bool ranked;            // ... ranked: by their rank, the first `rem` of them
  unsigned int rem;
  unsigned int bin_lo, bin_span;  // verify: keys that lie here must equal T
  bool verify;
};

// Draws chunks of THREADS * U entries by ticket until there are none left and writes their survivors.  fetch(run,
// run_end, v, idx): values and indices of entries run .. run_end - 1 of `total`, for a warp.  first: the block's first
// ticket; finished: chunks it has done.  False: a wait ran out.  other_keys: a key that `verify` rules out was seen.
template <int U, class Fetch>
__device__ __forceinline__ bool emit_chunks(const FinalizeParams& p, EmitShared& sh, const Choice& how, unsigned int total, unsigned int first,
                                            unsigned int* tickets, bool take_out, bool& other_keys, unsigned int& finished, Fetch&& fetch) {
  constexpr int THREADS = kEmitThreads, NW = THREADS / 32;
  constexpr unsigned int kChunk = THREADS * U, FULL = 0xFFFFFFFFu;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned int lt = (1u << lane) - 1u;
  const unsigned int k = (unsigned int)p.k, rem = how.rem;
  const unsigned int chunks = (total + kChunk - 1) / kChunk;
  uint32_t* out_idx = reinterpret_cast<uint32_t*>(p.payload + p.P.idx_off);
  unsigned int c = first;
  for (int turn = 0; c < chunks; turn ^= 1) {
    // ---------------- load, count ----------------
    const unsigned int run = c * kChunk + warp * (32 * U), run_end = min(total, run + 32 * U);
    uint32_t v[U], idx[U];
    unsigned int bs[U], bt[U], n_sure = 0, n_tied = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = idx[u] = bs[u] = bt[u] = 0;
    if (run < total) {
      fetch(run, run_end, v, idx);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t key = v[u] & 0x7FFFFFFFu;
        const bool live = run + u * 32 + lane < run_end;
        if (how.ranked) {
          bs[u] = __ballot_sync(FULL, live && key > how.T);
          bt[u] = __ballot_sync(FULL, live && key == how.T);
          n_tied += __popc(bt[u]);
          if (how.verify) other_keys |= live && key != how.T && key - how.bin_lo < how.bin_span;
        } else {
          bs[u] = __ballot_sync(FULL, live && (key > how.T || (key == how.T && idx[u] <= how.last_idx)));
        }
        n_sure += __popc(bs[u]);
      }
    }
    if (lane == 0) sh.warp_sum[warp] = make_uint2(n_sure, n_tied);
    __syncthreads();
    const uint2 ws = lane < NW ? sh.warp_sum[lane] : make_uint2(0u, 0u);
    const unsigned int sure_in_warps = __reduce_add_sync(FULL, lane < warp ? ws.x : 0u), chunk_sure = __reduce_add_sync(FULL, ws.x);
    unsigned int tied_in_warps = 0, chunk_tied = 0;
    if (how.ranked) {
      tied_in_warps = __reduce_add_sync(FULL, lane < warp ? ws.y : 0u);
      chunk_tied = __reduce_add_sync(FULL, ws.y);
    }
    const unsigned long long chunk_sum = ((unsigned long long)chunk_sure << 31) | chunk_tied;
    if (t == 0) {
      publish_sum(p.list.chunk_sum[0] + c, chunk_sum);
      sh.ticket[turn] = atomicAdd(tickets, 1u);
    }
    // ---------------- survivors before the chunk ----------------
    // the sums of up to 511 chunks before this one, and what comes before those from the 512th: thread t looks back t + 1
    unsigned long long back = 0;
    if ((unsigned)t < c) {
      back = wait_sum(t == THREADS - 1 ? p.list.chunk_sum[1] + (c - THREADS) : p.list.chunk_sum[0] + (c - 1 - t));
      if (back == 0) set_status(&p.ctl->status, NSML_ERR_TIMEOUT);
      back = back == 0 ? ~0ull : back & ~(1ull << 63);
    }
    const bool gave_up = __any_sync(FULL, back == ~0ull);
    const unsigned int back_sure = __reduce_add_sync(FULL, sure_of(back)), back_tied = how.ranked ? __reduce_add_sync(FULL, tied_of(back)) : 0u;
    if (lane == 0) sh.back_sum[warp] = make_uint2(back_sure, gave_up ? ~0u : back_tied);
    __syncthreads();
    const uint2 bw = lane < NW ? sh.back_sum[lane] : make_uint2(0u, 0u);
    if (__any_sync(FULL, bw.y == ~0u)) return false;  // (uniform over the block; the chunks behind this one time out as well)
    const unsigned int sure_before = __reduce_add_sync(FULL, bw.x), tied_before = how.ranked ? __reduce_add_sync(FULL, bw.y) : 0u;
    const unsigned long long upto = (((unsigned long long)sure_before << 31) | tied_before) + chunk_sum;
    if (t == 0) publish_sum(p.list.chunk_sum[1] + c, upto);
    const unsigned int p0 = sure_before + min(tied_before, rem);
    const unsigned int p1 = sure_of(upto) + min(tied_of(upto), rem);
    if (c == chunks - 1 && p1 != k && t == 0 && !how.verify) set_status(&p.ctl->status, NSML_ERR_INTERNAL);
    // The next kernel of the stream may be placed, to wait there: not earlier than hides its launch, because its blocks hold
    // what other streams' kernels could use.  (From the kernel's start on, eight streams that compress and sum 6.55M elements
    // take 22.5 us a pair of calls, now 18.4, 25M 59.0 and 55.3; a call by itself is the same.)
    pdl_launch_dependents();
    // ---------------- write the survivors ----------------
    unsigned int sure = sure_before + sure_in_warps, tied = tied_before + tied_in_warps;
    const bool int8 = p.bits == NSML_BITS_INT8;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const unsigned int s_mine = sure + __popc(bs[u] & lt), t_mine = tied + __popc(bt[u] & lt);
      if (((bs[u] >> lane) & 1u) || (((bt[u] >> lane) & 1u) && t_mine < rem)) {
        const unsigned int at = s_mine + min(t_mine, rem);
        if (at < k) {
          out_idx[at] = idx[u];
          if (int8) {
            sh.kept.val[at - p0] = v[u];
            sh.kept.idx[at - p0] = idx[u];
          } else {
            put_value(p, at, v[u]);
            if (take_out && v[u] != 0) p.residual[idx[u]] = not_carried(p, v[u]);  // (+0.0: see not_carried)
          }
        }
      }
      sure += __popc(bs[u]);
      tied += __popc(bt[u]);
    }
    // ---------------- int8: quantise ----------------
    if (int8 && p1 > p0 && p1 <= k) {  // uniform over the block
      const unsigned int qa = p0 / NSML_QBLOCK, qz = (p1 - 1) / NSML_QBLOCK;  // payload blocks the chunk has a part of
      auto q_end = [&](unsigned int q) { return min(k, (q + 1) * NSML_QBLOCK); };
      // shared with other chunks: the first if it starts before p0 or ends behind p1, the last if it ends behind p1
      const bool first_shared = qa * NSML_QBLOCK < p0 || q_end(qa) > p1, last_shared = qz != qa && q_end(qz) > p1;
      const bool shares = first_shared || last_shared;
      __syncthreads();  // sh.kept is complete
      auto park = [&](unsigned int q) {
        const unsigned int a = max(p0, q * NSML_QBLOCK), z = min(p1, q_end(q));
        for (unsigned int j = a + t; j < z; j += THREADS) p.raw_val[j] = __uint_as_float(sh.kept.val[j - p0]);
      };
      if (first_shared) park(qa);
      if (last_shared) park(qz);
      const unsigned int own_a = first_shared ? qa + 1 : qa, own_z = last_shared ? qz : qz + 1;
      if (shares) {
        __threadfence();
        __syncthreads();
        if (t < 2) {
          sh.done[t] = FULL;
          if (t == 0 ? first_shared : last_shared) {
            const unsigned int q = t == 0 ? qa : qz;
            const unsigned int mine = min(p1, q_end(q)) - max(p0, q * NSML_QBLOCK);
            if (atomicAdd(p.list.block_fill + q, mine) + mine == q_end(q) - q * NSML_QBLOCK) sh.done[t] = q;  // the last part
          }
        }
      }
      // inside the chunk: at most four
      if (own_a < own_z) {
        const unsigned int q = own_a + (warp >> 2);
        quantize_group(p, take_out ? p.residual : nullptr, sh.qmax, q, q < own_z, q < own_z ? q_end(q) - q * NSML_QBLOCK : 0u,
                       [&](unsigned int j) { return __uint_as_float(sh.kept.val[q * NSML_QBLOCK + j - p0]); },
                       [&](unsigned int j) { return sh.kept.idx[q * NSML_QBLOCK + j - p0]; });
      }
      if (shares) {
        __syncthreads();
        if (sh.done[0] != FULL || sh.done[1] != FULL) {
          __threadfence();  // the other chunks' parts are visible
          const unsigned int q = (warp >> 2) < 2 ? sh.done[warp >> 2] : FULL;
          quantize_group(p, take_out ? p.residual : nullptr, sh.qmax, q, q != FULL, q != FULL ? q_end(q) - q * NSML_QBLOCK : 0u,
                         [&](unsigned int j) { return __ldcg(p.raw_val + (size_t)q * NSML_QBLOCK + j); },
                         [&](unsigned int j) { return __ldcg(out_idx + (size_t)q * NSML_QBLOCK + j); });
        }
      }
    }
    if (c == 0 && t == 0) write_header(p);
    __syncthreads();  // the next ticket is there; shared memory may be overwritten
    c = sh.ticket[turn];
    ++finished;
  }
  return true;
}

// Waits (bounded) until a counter has reached `target`; called by the whole block.
template <class SH>  // (with a word sh.done[0])
__device__ __forceinline__ bool wait_count(const unsigned int* at, unsigned int target, Ctl* ctl, SH& sh) {
  if (threadIdx.x == 0) {
    unsigned int ok = 0;
    for (int polls = 0; polls < kMaxPolls && !ok; ++polls) {
      unsigned int seen;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(at) : "memory");
      ok = seen >= target;
      if (!ok && polls > 64) __nanosleep(64);
    }
    if (!ok) set_status(&ctl->status, NSML_ERR_TIMEOUT);
    sh.done[0] = ok;
  }
  __syncthreads();
  const bool ok = sh.done[0] != 0;
  __syncthreads();
  return ok;
}

// A phase of the general select: blocks draw its units of work by ticket; it is over when all units are finished.
// Whoever waits has no unit left to do, and every unit that is not finished has been drawn by a running block, so the
// phases need no co-resident grid.
template <class SH, class Work, class Last>
__device__ __forceinline__ bool run_phase(Ctl* ctl, int phase, unsigned int units, SH& sh, Work&& work, Last&& last) {
  unsigned int mine = 0;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) sh.ticket[0] = atomicAdd(&ctl->drawn[phase], 1u);
    __syncthreads();
    const unsigned int u = sh.ticket[0];
    if (u >= units) break;
    work(u);
    ++mine;
  }
  __syncthreads();
  last();
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0 && mine) atomicAdd(&ctl->finished[phase], mine);
  return wait_count(&ctl->finished[phase], units, ctl, sh);
}

// residual[idx_j] <- residual[idx_j] - v'_j for every entry of the payload, once it is complete.
__device__ __noinline__ void take_out_all(const FinalizeParams& p, EmitShared& sh) {
  const uint32_t* idx = reinterpret_cast<const uint32_t*>(p.payload + p.P.idx_off);
  const unsigned char* val = p.payload + p.P.val_off;
  const float* scale = reinterpret_cast<const float*>(p.payload + p.P.scale_off);
  const unsigned int k = (unsigned int)p.k;
  run_phase(p.ctl, 0, (k + kEmitThreads - 1) / kEmitThreads, sh, [&](unsigned int unit) {
    const unsigned int j = unit * kEmitThreads + threadIdx.x;
    if (j >= k) return;
    float v;
    if (p.bits == NSML_BITS_INT8) v = decode_i8(*reinterpret_cast<const volatile signed char*>(val + j), __ldcg(scale + (j >> 10)));
    else if (p.bits == NSML_BITS_FP16) v = decode_f16(__ldcg(reinterpret_cast<const uint16_t*>(val) + j));
    else v = __ldcg(reinterpret_cast<const float*>(val) + j);
    float* at = p.residual + __ldcg(idx + j);
    *at = __fsub_rn(*at, v);
  }, [] {});
}

// What k_emit's scheme does not cover, by all its blocks: the threshold by up to three histograms, each of one bin of
// the one before, until a bin is one key; of the list, or, where that holds fewer than k candidates, of the bucket.
template <int VT>
__device__ __noinline__ void general_select(const BucketSrc<VT>& src, const FinalizeParams& p, EmitShared& sh) {
  constexpr int THREADS = kEmitThreads, U = kEmitPer;
  constexpr unsigned int kUnit = 8 * kChunk, kMinShift = min_bin_shift<VT>();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const bool from_list = sh.sc.total >= (unsigned int)p.k;
  const unsigned int total = from_list ? sh.sc.total : (unsigned int)p.n;
  auto fetch = [&](unsigned int run, unsigned int run_end, uint32_t (&v)[U], uint32_t (&idx)[U]) {
    if (from_list) {
      fetch_run<VT, U>(p.list, sh.sc.off, p.tiles, run, run_end, v, idx);
      return;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      idx[u] = run + u * 32 + lane;
      v[u] = idx[u] < run_end ? src.load1(idx[u]) : 0u;
    }
  };
  const Window win = make_window<VT>(p.ctl);
  unsigned int bin_lo = 0, bin_shift = 31, rem = (unsigned int)p.k;
  if (from_list && sh.sc.bin_count == 0) bin_lo = win.hi;  // the threshold lies above the window
  if (from_list && sh.sc.bin_count != 0) {
    bin_lo = win.lo + (sh.sc.bin << win.shift);
    bin_shift = win.shift;
    rem = sh.sc.rem;
  }
  const unsigned int units = (total + kUnit - 1) / kUnit;
  auto& f = sh.general;
  for (int level = 0; bin_shift > kMinShift; ++level) {
    const unsigned int shift = max(kMinShift, bin_shift > 12 ? bin_shift - 12 : 0u), span = 1u << bin_shift;
    __syncthreads();
    for (int b = t; b < kMaxBins; b += THREADS) f.hist[b] = 0;
    unsigned int* ghist = p.hist + level * kMaxBins;
    const bool ok = run_phase(p.ctl, level, units, sh, [&](unsigned int unit) {
      for (unsigned int i = 0; i < kUnit / kChunk; ++i) {
        const unsigned int run = unit * kUnit + i * (unsigned)kChunk + warp * (32 * U), run_end = min(total, run + 32 * U);
        if (run >= total) break;
        uint32_t v[U], idx[U];
        fetch(run, run_end, v, idx);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const unsigned int rel = (v[u] & 0x7FFFFFFFu) - bin_lo;
          const bool inside = run + u * 32 + lane < run_end && rel < span;
          const unsigned int who = __ballot_sync(0xFFFFFFFFu, inside);
          if (inside) {  // (lanes with equal bins add once: there may be a great many equal keys)
            const unsigned int same = __match_any_sync(who, rel >> shift);
            if ((same & ((1u << lane) - 1u)) == 0) atomicAdd(&f.hist[rel >> shift], (unsigned int)__popc(same));
          }
        }
      }
    }, [&] {
      for (int b = t; b < kMaxBins; b += THREADS)
        if (f.hist[b]) atomicAdd(ghist + b, f.hist[b]);
    });
    if (!ok) return;
    constexpr int PER = kMaxBins / THREADS;
    unsigned int own[PER];
#pragma unroll
    for (int b = 0; b < PER; ++b) own[b] = __ldcg(ghist + t * PER + b);
    find_digit_from_top<PER, THREADS>(own, rem, f.tot, f.out);
    bin_lo += f.out[0] << shift;
    rem = f.out[1];
    bin_shift = shift;
  }
  // (the counters of chunks and payload blocks may have been used already)
  const unsigned int counters = max((total + kChunk - 1) / kChunk, (unsigned int)((p.k + NSML_QBLOCK - 1) / NSML_QBLOCK));
  const bool ok = run_phase(p.ctl, 3, (counters + THREADS - 1) / THREADS, sh, [&](unsigned int unit) {
    const unsigned int c = unit * THREADS + t;
    if (c < counters) {
      p.list.chunk_sum[0][c] = p.list.chunk_sum[1][c] = 0;
      p.list.block_fill[c] = 0;
    }
  }, [] {});
  if (!ok) return;
  Choice how;
  how.T = (bin_lo + ((1u << kMinShift) - 1u)) & ~((1u << kMinShift) - 1u);
  how.last_idx = 0;
  how.ranked = true;
  how.rem = rem;
  how.bin_lo = how.bin_span = 0;
  how.verify = false;
  __syncthreads();
  if (t == 0) sh.ticket[0] = atomicAdd(&p.ctl->drawn[4], 1u);
  __syncthreads();
  const unsigned int first = sh.ticket[0];
  __syncthreads();
  bool none = false;
  unsigned int finished = 0;
  emit_chunks<U>(p, sh, how, total, first, &p.ctl->drawn[4], p.residual != nullptr, none, finished, fetch);
}

// U: candidates per thread of a chunk.
template <int VT, int U>
__global__ void __launch_bounds__(kEmitThreads, 2) k_emit(BucketSrc<VT> src, FinalizeParams p) {
  constexpr int THREADS = kEmitThreads;
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  extern __shared__ __align__(16) unsigned char s_raw[];
  EmitShared& sh = *reinterpret_cast<EmitShared*>(s_raw);
  const int t = threadIdx.x;
  pdl_wait();
  if (t == 0) {
    const unsigned int first = atomicAdd(&p.ctl->ticket, 1u);
    sh.ticket[0] = first;
  }
  const Window win = make_window<VT>(p.ctl);
  scan_list(p, (unsigned int)p.k, sh.sc);
  const unsigned int first = sh.ticket[0];

  // ---------------- the threshold ----------------
  const unsigned int total = sh.sc.total, rem = sh.sc.rem, bin_count = sh.sc.bin_count;
  Choice how;
  how.T = win.key_of(sh.sc.bin);
  how.last_idx = 0;
  how.ranked = win.single();  // the bin is one key: its ties are kept by their rank
  how.rem = rem;
  how.bin_lo = win.lo + (sh.sc.bin << win.shift);
  how.bin_span = 1u << win.shift;
  bool general = bin_count == 0;
  if (!general && !how.ranked) {
    const unsigned int listed = min(bin_count, p.list.bin_room);
    for (unsigned int e = t; e < listed; e += THREADS) sh.bin[e] = __ldcg(p.list.bins + (size_t)sh.sc.bin * p.list.bin_room + e);
    __syncthreads();
    if (bin_count > listed) {
      // Too many keys to have been kept: if those that were are equal (a quantised gradient), the others very likely
      // are, too; that is checked as the list is read.
      int equal = 1;
      for (unsigned int e = t; e < listed; e += THREADS) equal &= sh.bin[e].x == sh.bin[0].x;
      how.ranked = __syncthreads_and(equal);
      how.T = sh.bin[0].x;
      general = !how.ranked;
      __syncthreads();
    } else {
      // rank of every key, by 1 << split neighbouring threads each
      const int split = listed >= THREADS ? 0 : min(5, 31 - __clz(THREADS / listed));
      for (unsigned int base = 0; base < listed << split; base += THREADS) {
        const unsigned int e = (base + t) >> split;
        uint2 me = make_uint2(0u, 0u);
        unsigned int ahead = 0;
        if (e < listed) {
          me = sh.bin[e];
          for (unsigned int q = t & ((1 << split) - 1); q < listed; q += 1 << split) {
            const uint2 o = sh.bin[q];
            ahead += o.x > me.x || (o.x == me.x && o.y < me.y);
          }
        }
        for (int o = (1 << split) >> 1; o > 0; o >>= 1) ahead += __shfl_xor_sync(FULL, ahead, o);
        if (e < listed && ahead == rem - 1) {  // exactly one key: the last survivor
          sh.T = me.x;
          sh.last_idx = me.y;
        }
      }
      __syncthreads();
      how.T = sh.T;
      how.last_idx = sh.last_idx;
    }
  }
  if (general) {  // uniform over the grid
    general_select<VT>(src, p, sh);
    return;
  }
  // Where one key was assumed, every key of the bin is compared with it.
  how.verify = how.ranked && !(VT == NSML_BF16 && win.single());
  // (what the payload carries is taken out of the residual at once, unless the call may have to be done over)
  bool other_keys = false;
  unsigned int finished = 0;
  const bool ok = emit_chunks<U>(p, sh, how, total, first, &p.ctl->ticket, p.residual != nullptr && !how.verify, other_keys, finished,
                                 [&](unsigned int run, unsigned int run_end, uint32_t (&v)[U], uint32_t (&idx)[U]) {
                                   fetch_run<VT, U>(p.list, sh.sc.off, p.tiles, run, run_end, v, idx);
                                 });
  if (!ok || !how.verify) return;
  if (other_keys) p.ctl->fallback = 1;
  __threadfence();
  __syncthreads();
  if (t == 0 && finished) atomicAdd(&p.ctl->done, finished);
  if (!wait_count(&p.ctl->done, (total + THREADS * U - 1) / (THREADS * U), p.ctl, sh)) return;
  if (*reinterpret_cast<volatile unsigned int*>(&p.ctl->fallback) != 0) {
    general_select<VT>(src, p, sh);
  } else if (p.residual != nullptr) {
    take_out_all(p, sh);
  }
}

}  // namespace nsml
