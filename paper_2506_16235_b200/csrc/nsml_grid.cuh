// Bucket -> payload without a candidate list, in one cooperative kernel (Alg. 2 Steps
// 2-3: pruned gradients read as zero; keep the k largest |g|, ties by lower index), for
// calls that keep a large fraction of a bucket: the list would be about as large.
//
// The bucket is cut into segments of 16 KB that the blocks take cyclically (block b:
// segments b, b + G, ...; a round of all blocks is a row), so that all SMs read one
// compact, moving window of it and a tensor whose gradients are larger than others' is
// spread over all of them.  A warp owns a slice, a 32nd, of each of its block's segments.
// Slices with a key >= lo stay in shared memory as they are while there is room beside the
// tables and lists, which grow with the bucket (148 SMs, at 0.5: 26.7 MB for 6.5M float32
// elements, which is all of them, 22.7 for 20M, 11.6 for 64M; bfloat16 26.4 for 20M, 19.6 for
// 64M; LARGE 30.7); the others are read from the bucket once more when the survivors are
// written.  Phases, separated by grid barriers:
//   sample  the bounds lo and hi of the threshold (nsml_select.cuh), by 16 of the blocks;
//           meanwhile every block has its first loads in flight
//   stream  per slice: kept or not, its largest key, its number of keys >= hi; the keys of
//           the window [lo, hi) in a list of the warp's and in a histogram
//   count   the bin of the k-th largest key; its keys are exchanged, and how many keys
//           above it every segment has.  (The bin holds more keys than are exchanged:
//           another histogram, of the bin, until it is narrow enough or a single key,
//           whose ties are then counted per segment and kept up to the last one's index.)
//   place   the exact threshold, every slice's place in the payload; int8: the largest
//           magnitude of every 1024 survivors
//   write   indices and values; int8 behind one more barrier
// A sample that misled costs more rounds: a threshold above the window, a histogram of
// what lies there; fewer than k candidates, a second stream with lo = 0.  A sample with
// fewer non-zero keys than its ranks says that the threshold is zero: the keys above it
// are counted in the stream, the others are ties, and there is no window.
// LARGE: tables and lists lie in the workspace (grid_plan says when), so that no bucket is too
// large: 200M float32 elements at 0.5 take 1.19 ms, 310M 1.8 (the candidate list, which
// took such calls for a while, 2.8 and 6.1; the radix select before 1.72 and 2.7).
//
// What bounds it: instructions, about 580 per 128 elements at 0.5 by the counters, the
// walk that writes the survivors and the stream before all, and four or five steps in which every block waits for the
// others (2 to 4 us each).  Measured (one B200, whole call, before / now; before: a radix
// select in three digits over a shared-memory copy, every element looked at by every
// phase, add and subtract of a residual as kernels of their own): 6.55M float32 elements
// at 0.5 as int8 72 / 57 us, 64M at 0.5 582 / 332, 67M bfloat16 at 0.5 as fp16 619 / 175,
// 25M with a residual at 0.5 357 / 190.  In the kernel, 6.55M at 0.5: bounds known at 11
// us, streamed 20, bin 25, places 31, maxima 35, written 48-52.
// Tried on the way: lists of candidates instead of slices (65 instructions per 32
// entries and phase: 70 us), maxima and codes in two walks over the slices (58), one walk
// per phase over all kept slices (51 in the kernel where it takes 50 now, and 357 us
// instead of 332 at 64M), 512 threads twice per SM (3-4 us more in the shared steps).
#pragma once

#include <type_traits>

#include "nsml_finalize.cuh"

namespace nsml {

constexpr int kGridSamplers = kSamples / kGridThreads;  // blocks that take the sample, a stratum per thread
constexpr unsigned int kGridMembers = 2048;  // keys of the threshold's bin that are exchanged
// The window's histogram.  Adds to one global address run at one per nanosecond, and the keys of a bin may be any number (a
// repeated value; a window from zero on): a block counts in shared memory and adds a bin's count once.  (With an add per
// key, 25M float32 elements of which 54 % are zero took 18 ms at 0.5, now 0.12; of one value 16, now 0.20.)  In a short
// float32 bucket, whose window has a few keys per warp and most bins fewer than kGridDirect per block, those few are added
// at once and the pass over the bins behind them is left out; lists of kGridShareCap and more entries pay for it.  us, pass
// left out / not: 6.55M at 0.5 57.2 / 58.2, 12M 80.8 / 79.1, 25M 150 / 142.
constexpr unsigned int kGridFewBins = 256, kGridShareCap = 128;
constexpr unsigned int kGridDirect = 4;                // a bin's first keys, counted in the upper three bits of its word, too
constexpr unsigned int kGridCounted = (1u << 29) - 1;  // all its keys

struct GridShared {
  union {
    unsigned int hist[kMaxBins];
    uint4 slice[kGridWarps][32];         // a slice that is not kept, while its survivors are written
  };
  unsigned char stage[kGridWarps][256];  // offsets of a slice's survivors
  unsigned long long listed;  // candidates << 32 | those above the window
  unsigned int tot[kGridWarps], out[3];
  unsigned int lo, hi, pool;
  unsigned int zeros, heavy;  // zeros among the keys counted; bins hold keys that have not been added to the grid's
  int ok;
};
static_assert(sizeof(GridShared) == kGridSharedBytes, "the plan counts on it");
// The sample counts keys by their top 15 bits (of bfloat16: all), those of 64 octaves from 2^-49 on, all smaller ones that
// are not zero in its first bin.
constexpr unsigned int kGridSampleBins = 8192, kGridSampleBase = 78u << 7;

struct SliceScale { float scale, inv; unsigned int slots; bool one; };  // one: the slice's survivors share a payload block

template <int DTYPE, bool FEEDBACK, bool MASKED, bool LARGE>
__global__ void __launch_bounds__(kGridThreads, 1)
k_select_grid(BucketSrc<DTYPE> src, FinalizeParams p, unsigned int segs, unsigned int rows, unsigned int cap, unsigned int room,
              unsigned int rank_lo, unsigned int rank_hi) {
  constexpr int VT = FEEDBACK ? NSML_F32 : DTYPE;  // what the list holds
  constexpr bool PACKED = VT == NSML_BF16;         // slices hold bfloat16 values
  constexpr bool SHORT = PACKED && !LARGE;         // list entries are bfloat16 keys << 16 | place
  using Place = typename std::conditional<LARGE, unsigned int, unsigned short>::type;  // an entry's: row and offset in its slice
  constexpr int ESIZE = DTYPE == NSML_F32 ? 4 : 2;
  constexpr int EPL = FEEDBACK ? 4 : 16 / ESIZE;   // elements of a lane's load
  constexpr unsigned int SEG = grid_seg<VT>(), SLICE = SEG / kGridWarps;  // elements of a segment, of a warp's part
  constexpr int OFF_BITS = grid_off_bits<VT>();
  constexpr unsigned int SLOTS = grid_slots<VT>();
  static_assert(SEG == kGridThreads * EPL && SLICE == 1u << OFF_BITS, "a lane has EPL elements of a segment");
  constexpr unsigned int UNIT = VT == NSML_BF16 ? 65536u : 1u;  // the smallest key that is not zero; keys are multiples of it
  constexpr int DEPTH = FEEDBACK ? 4 : 6;  // rows whose loads are in flight
  constexpr int PAIR = 2;                  // rows that are looked at together
  constexpr int THREADS = kGridThreads, NW = kGridWarps, PITCH = kGridPitch;
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  extern __shared__ __align__(16) unsigned char s_raw[];
  GridShared& sh = *reinterpret_cast<GridShared*>(s_raw);
  // per row and warp: survivors | ties << 16; place of the slice's first survivor; largest key
  unsigned char* tables = LARGE ? reinterpret_cast<unsigned char*>(p.list.off) + blockIdx.x * grid_table_bytes<VT>(rows) : s_raw + sizeof(GridShared);
  unsigned int* cnt = reinterpret_cast<unsigned int*>(tables);
  unsigned int* base = cnt + rows * PITCH;
  unsigned int* top = base + rows * PITCH;
  unsigned int* row_s = top + rows * PITCH;     // per row: survivors, ties; those in the segments before the block's
  unsigned int* row_t = row_s + rows;
  unsigned int* part_s = row_t + rows;
  unsigned int* part_t = part_s + rows;
  unsigned int* extra = part_t + rows;          // survivors of the threshold's bin before the block's segment
  unsigned int* row_at = extra + rows;          // place of the segment's first survivor
  unsigned int* qm = row_at + rows;             // [rows][SLOTS]: largest magnitude, then scale, of the payload blocks
  unsigned int* qi = qm + rows * SLOTS;         // their inverses
  unsigned short* kept = reinterpret_cast<unsigned short*>(qi + rows * SLOTS) + (threadIdx.x >> 5) * rows;  // [NW][rows]: the slice's place + 1
  constexpr unsigned int kNotHere = 0xFFFFu;    // ... it is to be read from the bucket
  unsigned char* lists = s_raw + sizeof(GridShared) + (size_t)rows * grid_row_bytes<VT>();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned int lt = (1u << lane) - 1u, G = gridDim.x, blk = blockIdx.x;
  const unsigned int n = (unsigned int)p.n, k = (unsigned int)p.k;
  const size_t list = LARGE ? ((size_t)blk * NW + warp) * cap : warp * cap;  // the warp's list: keys, and places in its part
  uint32_t* s_val = (LARGE ? p.list.val : reinterpret_cast<uint32_t*>(lists)) + list;
  Place* s_pos = (LARGE ? reinterpret_cast<Place*>(p.raw_val) : reinterpret_cast<Place*>(lists + (size_t)NW * cap * 4)) + (SHORT ? 0 : list);
  uint4* s_slice = reinterpret_cast<uint4*>(s_raw + grid_smem<VT>(LARGE ? 0 : rows, LARGE ? 0 : cap, 0));  // the block's slices
  float* residual = p.residual;
  unsigned int barriers = 0;

  // ---------------- the first loads ----------------
  constexpr int KEYS = sample_keys<DTYPE>();
  const bool sampler = rank_lo != 0 && blk < (unsigned)kGridSamplers;
  uint4 sampled = make_uint4(0u, 0u, 0u, 0u);
  float4 addend[KEYS / 4];
  uint32_t sample_mask = 0;
  if (sampler) {  // (the keys that k_sample reads)
    const unsigned long long stratum = (unsigned long long)blk * THREADS + t;
    const unsigned long long begin = stratum * n / kSamples, end = (stratum + 1) * n / kSamples;
    unsigned long long pos = (begin + mix32((uint32_t)stratum * 0x9E3779B1u + 0x85EBCA6Bu) % (uint32_t)(end - begin)) & ~(unsigned long long)(KEYS - 1);
    if (pos + KEYS > n) pos = (n - KEYS) & ~(unsigned long long)(KEYS - 1);
    sampled = __ldcs(reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(src.grad) + pos * ESIZE));
#pragma unroll
    for (int e = 0; e < KEYS; e += 4)
      if (FEEDBACK) addend[e / 4] = *reinterpret_cast<const float4*>(residual + pos + e);
    if (MASKED) sample_mask = __ldg(src.mask + (pos >> 5)) >> (unsigned)(pos & 31);
  }
  // a row's loads: those of whole segments
  const unsigned int whole_segs = n / SEG, full = blk < whole_segs ? (whole_segs - blk - 1) / G + 1 : 0u;
  const unsigned int stride = G * SEG, mine0 = blk * SEG + warp * SLICE + lane * EPL;  // the lane's first element of row 0
  uint4 q[DEPTH];
  float4 res[FEEDBACK ? DEPTH : 1];
  uint32_t mw[MASKED ? DEPTH : 1];
  auto load = [&](int slot, unsigned int i) {  // elements i ...
    const unsigned char* g = static_cast<const unsigned char*>(src.grad) + (size_t)i * ESIZE;
    if (EPL * ESIZE == 16) {
      q[slot] = __ldcs(reinterpret_cast<const uint4*>(g));
    } else {
      const uint2 v = __ldcs(reinterpret_cast<const uint2*>(g));
      q[slot] = make_uint4(v.x, v.y, 0u, 0u);
    }
    if (FEEDBACK) res[FEEDBACK ? slot : 0] = *reinterpret_cast<const float4*>(residual + i);
    if (MASKED) mw[MASKED ? slot : 0] = __ldg(src.mask + (i >> 5));
  };
  auto load_first = [&]() {
#pragma unroll
    for (int d = 0; d < DEPTH; ++d)
      if (d < (int)full) load(d, mine0 + d * stride);
  };
  if (!sampler) load_first();

  // ---------------- the sample ----------------
  for (unsigned int i = t; i < kMaxBins; i += THREADS) sh.hist[i] = 0;
  for (unsigned int i = t; i < rows * SLOTS; i += THREADS) qm[i] = 0;
  for (unsigned int i = t; i < rows; i += THREADS) extra[i] = row_t[i] = part_t[i] = 0;
  if (t == 0) sh.lo = sh.hi = sh.pool = sh.zeros = sh.heavy = 0, sh.listed = 0;
  __syncthreads();
  if (sampler) {
    uint32_t b[KEYS];
    unpack16<DTYPE, KEYS>(sampled, b);
#pragma unroll
    for (int e = 0; e < KEYS; ++e) {
      if (FEEDBACK) b[e] = __float_as_uint(__fadd_rn(__uint_as_float(b[e]), reinterpret_cast<const float*>(addend)[e]));
      if (MASKED && ((sample_mask >> e) & 1u)) b[e] = 0;
      const unsigned int key = b[e] & 0x7FFFFFFFu, bin = min(max(key >> 16, kGridSampleBase) - kGridSampleBase, kGridSampleBins - 1);
      if (key != 0) atomicAdd(&sh.hist[bin >> 1], 1u << (16 * (bin & 1)));  // (a block has at most 8192 keys)
    }
  }
  pdl_wait();  // the control block and the histograms are cleared
  pdl_launch_dependents();
  unsigned int* qmax = reinterpret_cast<unsigned int*>(p.list.chunk_sum[0]);
  if (p.bits == NSML_BITS_INT8)
    for (unsigned long long i = (unsigned long long)blk * THREADS + t; i < p.P.nblocks; i += (unsigned long long)G * THREADS) qmax[i] = 0;
  if (rank_lo != 0) {
    unsigned int* shist = p.list.group_count;
    if (sampler) {
      __syncthreads();
      for (int b = t; b < kMaxBins; b += THREADS)
        if (sh.hist[b]) {
          const unsigned int two = sh.hist[b];
          if (two & 0xFFFFu) atomicAdd(shist + 2 * b, two & 0xFFFFu);
          if (two >> 16) atomicAdd(shist + 2 * b + 1, two >> 16);
          sh.hist[b] = 0;
        }
      load_first();  // (behind the sample, which the other blocks wait for)
    }
    __syncthreads();
    // as grid_barrier, but only the samplers arrive
    if (t == 0) {
      if (sampler) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&p.ctl->sampled), "r"(1u) : "memory");
      int ok = 0;
      for (int polls = 0; polls < kMaxPolls && !ok; ++polls) {
        unsigned int seen;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&p.ctl->sampled) : "memory");
        ok = seen >= (unsigned)kGridSamplers;
        if (polls > 256) __nanosleep(64);
      }
      if (!ok) set_status(&p.ctl->status, NSML_ERR_TIMEOUT);
      sh.ok = ok;
    }
    __syncthreads();
    if (!sh.ok) return;
    constexpr int PER = kGridSampleBins / THREADS;
    unsigned int own[PER], mine = 0;
#pragma unroll
    for (int b = 0; b < PER; b += 4) {
      const uint4 v = __ldcg(reinterpret_cast<const uint4*>(shist + t * PER + b));
      own[b] = v.x; own[b + 1] = v.y; own[b + 2] = v.z; own[b + 3] = v.w;
    }
#pragma unroll
    for (int b = 0; b < PER; ++b) mine += own[b];
    unsigned int incl = mine;  // this thread and all higher lanes of the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int v = __shfl_down_sync(FULL, incl, o);
      if (lane + o < 32) incl += v;
    }
    if (lane == 0) sh.tot[warp] = incl;
    __syncthreads();
    unsigned int above = incl - mine + __reduce_add_sync(FULL, lane > warp && lane < NW ? sh.tot[lane] : 0u);
#pragma unroll
    for (int b = PER - 1; b >= 0; --b) {
      const unsigned int bin = t * PER + b;
      if (above < rank_lo && rank_lo <= above + own[b]) sh.lo = bin == 0 ? UNIT : (bin + kGridSampleBase) << 16;
      if (above < rank_hi && rank_hi <= above + own[b]) sh.hi = bin + 1 < kGridSampleBins ? (bin + 1 + kGridSampleBase) << 16 : 0x80000000u;
      above += own[b];
    }
    __syncthreads();
  }
  unsigned int lo = min(sh.lo, kInfKey), hi = sh.hi;  // (as make_window)
  // The sample holds fewer keys that are not zero than either rank, or everything is kept and there was no sample: the
  // threshold is taken for zero, with no window; the number of other keys will tell.
  auto all_sure = [&]() { return (sh.lo | sh.hi) == 0; };
  if (all_sure()) hi = lo = UNIT;
  else if (hi <= lo) hi = 0x80000000u;

  // ---------------- what a warp keeps ----------------
  unsigned int len = 0;  // keys inside the window; more than cap: they are not all in the list
  auto row_index = [&](unsigned int row) { return row * stride + blk * SEG + warp * SLICE; };  // the slice's first element
  // unpacks a lane's elements and applies its mask bits
  auto unpack = [&](const uint4& w, uint32_t m, uint32_t (&bits)[EPL]) {
    unpack16<VT, EPL>(w, bits);
    if (MASKED) {
#pragma unroll
      for (int e = 0; e < EPL; ++e)
        if (m & (1u << e)) bits[e] = 0;
    }
  };
  auto pack = [&](const uint32_t (&bits)[EPL]) {
    if (PACKED) return make_uint4(bits[0] >> 16 | bits[1], bits[2] >> 16 | bits[3], bits[4 % EPL] >> 16 | bits[5 % EPL], bits[6 % EPL] >> 16 | bits[7 % EPL]);
    return make_uint4(bits[0], bits[1], bits[2], bits[3]);
  };
  // of a lane's elements in a slice: the number before them in lower lanes, and in all
  auto lanes_before = [&](unsigned int mine, unsigned int& all) {
    unsigned int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int up = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += up;
    }
    all = __shfl_sync(FULL, incl, 31);
    return incl - mine;
  };
  // Calls f(row, bits, here, at) for the slices that may hold candidates and are wanted(row), in order, by all lanes: a
  // lane's EPL elements from offset lane * EPL on, of which the first `here` exist; where the slice is kept.
  auto walk_slices = [&](auto&& wanted, auto&& f) {
    for (unsigned int r0 = 0; r0 < rows; r0 += 32) {
      const unsigned int mine = r0 + lane < rows && wanted(r0 + lane) ? kept[r0 + lane] : 0u;
      unsigned int left = __ballot_sync(FULL, mine != 0);
      uint4 w = make_uint4(0u, 0u, 0u, 0u);
      uint32_t m = 0;
      unsigned int row = 0, at = 0;
      auto fetch = [&]() {  // the first of what is left
        const int r = __ffs(left) - 1;
        row = r0 + r;
        at = __shfl_sync(FULL, mine, r);
        m = 0;
        if (at != kNotHere) {
          w = s_slice[(at - 1) * 32 + lane];
        } else if (row_index(row) + SLICE <= n) {
          const unsigned int i = row_index(row) + lane * EPL;
          if (FEEDBACK) w = *reinterpret_cast<const uint4*>(residual + i);
          else w = *reinterpret_cast<const uint4*>(static_cast<const unsigned char*>(src.grad) + (size_t)i * ESIZE);
          if (MASKED) m = src.mask[i >> 5] >> (i & 31);
        }
      };
      if (left != 0) fetch();
      while (left != 0) {
        const unsigned int this_row = row, this_at = at, i = row_index(row) + lane * EPL;
        uint32_t bits[EPL];
        unpack(w, m, bits);
        left &= left - 1;
        if (left != 0) fetch();  // the next one's load is in flight while this one is worked on
        int here = EPL;
        if (row_index(this_row) + SLICE > n) {
          here = i < n ? min((int)(n - i), EPL) : 0;
          if (this_at == kNotHere) {
#pragma unroll
            for (int e = 0; e < EPL; ++e)
              bits[e] = e >= here || (MASKED && src.pruned(i + e)) ? 0u : FEEDBACK ? __float_as_uint(residual[i + e]) : src.raw1(i + e);
          }
        }
        f(this_row, bits, here, this_at);
      }
    }
  };
  auto all_slices = [](unsigned int) { return true; };
  // Calls f(live, row, key, offset) for the list, in order, by all lanes.
  auto walk_list = [&](auto&& f) {
#pragma unroll 1
    for (unsigned int i = lane; i - lane < len; i += 32) {
      const uint32_t v = i < len ? s_val[i] : 0u;
      const unsigned int pos = SHORT ? v & 0xFFFFu : i < len ? s_pos[SHORT ? 0 : i] : 0u;
      f(i < len, pos >> OFF_BITS, SHORT ? v & 0xFFFF0000u : v, pos & (SLICE - 1));
    }
  };

  // ---------------- stream; the threshold's bin ----------------
  unsigned int wlo = lo, whi = hi, shift = 0;
  auto set_window = [&](unsigned int from, unsigned int to) {
    wlo = from;
    whi = to;
    shift = 32 - __clz((whi - wlo - 1) / kMaxBins);
    if (VT == NSML_BF16) shift = max(shift, 16u);
  };
  set_window(lo, hi);
  if (all_sure()) lo = 0;
  unsigned int rem = k, in_bin = 0;
  bool single = false, zero = false;     // the bin is one key; that is zero, and all other keys have been counted
  bool again = false, streaming = true;  // the stream is repeated, with lo = 0; it is still to be done
  unsigned int above = 0;                // of the lane: keys above the window
  bool nonfinite = false;
  // keeps a slice, mask bits applied, of which the first `here` elements of a lane exist
  auto keep_slice = [&](const uint32_t (&bits)[EPL], int here, unsigned int row) {
    unsigned int c = 0, inside = 0, most = 0, at = 0;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      const uint32_t key = bits[e] & 0x7FFFFFFFu;
      c += key >= whi;  // (missing ones are zeros)
      inside |= (unsigned)(key - wlo < whi - wlo) << e;
      most = max(most, key);
    }
    if (here < EPL) inside &= (1u << here) - 1u;
    above += c;
    c = __reduce_add_sync(FULL, c);
    most = __reduce_max_sync(FULL, most);
    nonfinite |= most >= kInfKey;
    if (lane == 0) {
      cnt[row * PITCH + warp] = c;
      top[row * PITCH + warp] = most;
      at = atomicAdd(&sh.pool, 1u);
      kept[row] = at < room ? (unsigned short)(at + 1) : (unsigned short)kNotHere;
    }
    at = __shfl_sync(FULL, at, 0);
    if (at < room) s_slice[at * 32 + lane] = pack(bits);
    const unsigned int any = __ballot_sync(FULL, inside != 0);
    if (any == 0) return;
    unsigned int rank = __popc(any & lt), all = __popc(any);
    if (__any_sync(FULL, (inside & (inside - 1)) != 0)) rank = lanes_before(__popc(inside), all);
    if (len + all <= cap) {
      rank += len;
#pragma unroll
      for (int e = 0; e < EPL; ++e)
        if (inside & (1u << e)) {
          const unsigned int pos = row << OFF_BITS | (lane * EPL + e);
          s_val[rank] = SHORT ? (bits[e] & 0x7FFF0000u) | pos : bits[e] & 0x7FFFFFFFu;
          if (!SHORT) s_pos[rank] = (Place)pos;
          ++rank;
        }
    }
    len += all;
  };
  for (int level = 0;; ++level) {  // (at most four: what lies beyond the window, then 12 + 12 + 7 bits of it)
    if (streaming) {
      len = 0;
      for (unsigned int row = lane; row < rows; row += 32) {
        kept[row] = 0;
        cnt[row * PITCH + warp] = 0;
      }
      __syncwarp();
      for (unsigned int row0 = 0; row0 < full; row0 += DEPTH) {
#pragma unroll
        for (int d = 0; d < DEPTH; d += PAIR) {
          const unsigned int row = row0 + d;
          if (row >= full) break;
          uint4 w[PAIR];
          uint32_t m2[PAIR], top[PAIR];
#pragma unroll
          for (int h = 0; h < PAIR; ++h) {
            const unsigned int i = mine0 + (row + h) * stride;
            top[h] = 0;
            if (row + h >= full) continue;
            w[h] = q[d + h];
            if (FEEDBACK) {
              uint32_t b[4];
              if (DTYPE == NSML_F32) {
                b[0] = w[h].x; b[1] = w[h].y; b[2] = w[h].z; b[3] = w[h].w;
              } else {
                b[0] = w[h].x << 16; b[1] = w[h].x & 0xFFFF0000u;
                b[2] = w[h].y << 16; b[3] = w[h].y & 0xFFFF0000u;
              }
              float4 s = res[FEEDBACK ? d + h : 0];
              if (!again) {  // (repeated: the residual holds the sum already)
                s = make_float4(__fadd_rn(__uint_as_float(b[0]), s.x), __fadd_rn(__uint_as_float(b[1]), s.y),
                                __fadd_rn(__uint_as_float(b[2]), s.z), __fadd_rn(__uint_as_float(b[3]), s.w));
                *reinterpret_cast<float4*>(residual + i) = s;
              }
              w[h] = make_uint4(__float_as_uint(s.x), __float_as_uint(s.y), __float_as_uint(s.z), __float_as_uint(s.w));
            }
            m2[h] = mw[MASKED ? d + h : 0];
            if (row + h + DEPTH < full) load(d + h, i + DEPTH * stride);
            // the largest key
            if (PACKED) {
              const uint32_t m = __vmaxu2(__vmaxu2(w[h].x & 0x7FFF7FFFu, w[h].y & 0x7FFF7FFFu), __vmaxu2(w[h].z & 0x7FFF7FFFu, w[h].w & 0x7FFF7FFFu));
              top[h] = max(m & 0xFFFF0000u, m << 16);
            } else {
              top[h] = max(max(w[h].x & 0x7FFFFFFFu, w[h].y & 0x7FFFFFFFu), max(w[h].z & 0x7FFFFFFFu, w[h].w & 0x7FFFFFFFu));
            }
          }
          // usually nothing is kept of a slice
          if (!__any_sync(FULL, (PAIR == 2 ? max(top[0], top[PAIR - 1]) : top[0]) >= lo)) continue;
#pragma unroll
          for (int h = 0; h < PAIR; ++h) {
            if (row + h >= full) break;
            if (PAIR > 1 && !__any_sync(FULL, top[h] >= lo)) continue;
            uint32_t bits[EPL];
            unpack(w[h], m2[h] >> (unsigned)((lane * EPL) & 31), bits);
            keep_slice(bits, EPL, row + h);
          }
        }
      }
      if (full < rows && full * G + blk < segs) {  // the bucket's ragged end
        uint32_t bits[EPL];
        int here = 0;
#pragma unroll
        for (int e = 0; e < EPL; ++e) {
          const unsigned int i = mine0 + full * stride + e;
          bits[e] = 0;
          if (i >= n) continue;
          ++here;
          if (FEEDBACK) {
            float s = residual[i];
            if (!again) {
              s = __fadd_rn(__uint_as_float(src.raw1(i)), s);
              residual[i] = s;
            }
            bits[e] = __float_as_uint(s);
          } else {
            bits[e] = src.raw1(i);
          }
          if (MASKED && src.pruned(i)) bits[e] = 0;
        }
        keep_slice(bits, here, full);
      }
      __syncwarp();
      streaming = false;
    }
    // ---------------- histogram of the window ----------------
    unsigned int* ghist = p.hist + level * kMaxBins;
    {
      const unsigned int direct = (whi - wlo - 1) >> shift < kGridFewBins || cap >= kGridShareCap ? 0u : kGridDirect;
      unsigned int zeros = 0;  // of the lane: a window from zero on may hold little else, so they are added together
      if (level != 0) {
        for (unsigned int b = t; b < kMaxBins; b += THREADS) sh.hist[b] = 0;
        __syncthreads();
      }
      if (len > cap) {
        walk_slices(all_slices, [&](unsigned int, const uint32_t (&bits)[EPL], int here, unsigned int) {
#pragma unroll
          for (int e = 0; e < EPL; ++e) {
            const uint32_t key = bits[e] & 0x7FFFFFFFu;
            if (e >= here || key - wlo >= whi - wlo) continue;
            if (key == 0) ++zeros;
            else atomicAdd(&sh.hist[(key - wlo) >> shift], 1u);
          }
        });
        if (!PACKED && lane == 0) sh.heavy = 1;
      } else {
        walk_list([&](bool live, unsigned int, uint32_t key, unsigned int) {
          if (live && key - wlo < whi - wlo) {
            const unsigned int bin = (key - wlo) >> shift;
            zeros += key == 0;
            if (PACKED) {
              atomicAdd(&sh.hist[bin], 1u);
            } else if ((atomicAdd(&sh.hist[bin], 1u) & kGridCounted) < direct) {
              atomicAdd(ghist + bin, 1u);
              atomicAdd(&sh.hist[bin], kGridCounted + 1u);
            } else {
              sh.heavy = 1;
            }
          }
        });
      }
      if (wlo == 0) {
        zeros = __reduce_add_sync(FULL, zeros);
        if (lane == 0 && zeros != 0) {
          if (len > cap) atomicAdd(&sh.hist[0], zeros);
          atomicAdd(&sh.zeros, zeros);
        }
      }
      if (level == 0) {
        const unsigned int sure = __reduce_add_sync(FULL, above);
        if (lane == 0 && sure + len != 0) atomicAdd(&sh.listed, (unsigned long long)(sure + len) << 32 | sure);
        if (nonfinite) set_status(&p.ctl->status, NSML_ERR_NONFINITE);
      }
      __syncthreads();
      if (level == 0 && t == 0) atomicAdd(&p.ctl->listed_above, sh.listed);
      if (t == 0 && sh.zeros != 0) {
        atomicAdd(&p.ctl->zeros[level], sh.zeros);
        sh.zeros = 0;
      }
      if (wlo != whi && (PACKED || sh.heavy)) {
        for (unsigned int b = t; b <= (whi - wlo - 1) >> shift; b += THREADS)
          if (const unsigned int c = (sh.hist[b] & kGridCounted) - (sh.hist[b] >> 29)) atomicAdd(ghist + b, c);
      }
    }
    if ((level == 1 || (lo == 0 && rank_lo != 0)) && blk == 0 && t == 0) p.ctl->drawn[3] = 1;  // (the sample was not enough)
    if (!grid_barrier(p.ctl, ++barriers * G, sh)) return;
    constexpr int PER = kMaxBins / THREADS;
    unsigned int own[PER];
#pragma unroll
    for (int b = 0; b < PER; b += 4) {
      const uint4 v = __ldcg(reinterpret_cast<const uint4*>(ghist + t * PER + b));
      own[b] = v.x; own[b + 1] = v.y; own[b + 2] = v.z; own[b + 3] = v.w;
    }
    if (level == 0) {  // (all decisions here are uniform over the grid)
      const unsigned long long both = __ldcg(&p.ctl->listed_above);
      const unsigned int listed = all_sure() ? n : (unsigned int)(both >> 32), higher = (unsigned int)both;
      if (listed < k) {  // the sample misled: keep everything; the threshold lies below lo
        rem = k - listed;
        set_window(0, lo);
        lo = 0;
        again = streaming = true;
        __syncthreads();
        if (t == 0) sh.pool = 0;
        __syncthreads();
        load_first();
        continue;
      }
      if (higher >= k && k != n) {  // the threshold lies above the window
        set_window(whi, 0x80000000u);
        len = cap + 1;  // (the list is of no use)
        continue;
      }
      rem = k - higher;
      if (all_sure()) {  // (rem of the zeros are kept: of k = n elements all, if there are any)
        set_window(0, UNIT);
        single = zero = true;
        break;
      }
    }
    find_digit_from_top<PER, THREADS>(own, rem, sh.tot, sh.out);
    const unsigned int from = wlo + (sh.out[0] << shift), width = 1u << shift;
    set_window(from, min(whi, from + width));
    rem = sh.out[1];
    in_bin = sh.out[2];
    if (from == 0) {
      const unsigned int larger = in_bin - __ldcg(&p.ctl->zeros[level]);
      if (rem > larger) {  // the threshold is zero
        set_window(0, UNIT);
        rem -= larger;
        single = true;
        break;
      }
    }
    if (width == UNIT) {
      single = true;  // one key: its ties are kept up to the last one's index
      break;
    }
    if (in_bin <= kGridMembers) break;
    if (level == 3) {  // (cannot be)
      set_status(&p.ctl->status, NSML_ERR_INTERNAL);
      return;
    }
  }

  // ---------------- keys above the bin per segment; the bin's keys ----------------
  auto exchange = [&](uint32_t key, unsigned int idx) {
    const unsigned int slot = atomicAdd(&p.ctl->members, 1u);
    if (slot < kGridMembers) p.list.bins[slot] = make_uint2(key, idx);
  };
  if (zero) {  // a slice's other elements are ties
    for (unsigned int row = lane; row < rows; row += 32)
      if (row_index(row) < n) cnt[row * PITCH + warp] |= (min(n - row_index(row), SLICE) - cnt[row * PITCH + warp]) << 16;
  } else if (len > cap) {
    walk_slices(all_slices, [&](unsigned int row, const uint32_t (&bits)[EPL], int here, unsigned int) {
      unsigned int c = 0;
#pragma unroll
      for (int e = 0; e < EPL; ++e) {
        const uint32_t key = bits[e] & 0x7FFFFFFFu;
        c += key >= whi;
        if (key - wlo < whi - wlo && e < here) {
          if (single) c += 1u << 16;
          else exchange(key, row_index(row) + lane * EPL + e);
        }
      }
      c = __reduce_add_sync(FULL, c);
      if (lane == 0) cnt[row * PITCH + warp] = c;
    });
  } else {  // the keys above the sampled window have been counted
    walk_list([&](bool live, unsigned int row, uint32_t key, unsigned int off) {
      if (!live) return;
      const bool inside = key - wlo < whi - wlo;
      if (key >= whi) atomicAdd(cnt + row * PITCH + warp, 1u);
      else if (inside && single) atomicAdd(cnt + row * PITCH + warp, 1u << 16);
      else if (inside) exchange(key, row_index(row) + off);
    });
  }
  __syncwarp();
  __syncthreads();
  unsigned short* seg_s = reinterpret_cast<unsigned short*>(p.list.tile_count);  // of a segment: survivors for certain, ties
  unsigned short* seg_t = reinterpret_cast<unsigned short*>(p.list.block_fill);
  for (unsigned int i = t; i < (rows * NW + 31) / 32 * 32; i += THREADS) {
    const unsigned int row = i / NW, seg = row * G + blk;
    const unsigned int mine = row < rows ? cnt[row * PITCH + i % NW] : 0u;
    unsigned int c = mine;  // of this and the lower warps
#pragma unroll
    for (int o = 1; o < NW; o <<= 1) {
      const unsigned int up = __shfl_up_sync(FULL, c, o, NW);
      if ((lane & (NW - 1)) >= o) c += up;
    }
    if (row < rows) base[row * PITCH + i % NW] = c - mine;
    if (i % NW == NW - 1 && row < rows && seg < segs) {
      seg_s[seg] = (unsigned short)c;
      if (single) seg_t[seg] = (unsigned short)(c >> 16);
    }
  }
  if (!grid_barrier(p.ctl, ++barriers * G, sh)) return;

  // ---------------- the threshold, every survivor's place ----------------
  static_assert(kGridMembers == 2 * THREADS, "two exchanged keys per thread");
  uint2 member[2] = {};  // (key, index)
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (!single && t + u * THREADS < in_bin) member[u] = __ldcg(p.list.bins + t + u * THREADS);
  {
    // A row's counts, and those before the block's segment, by a warp; two segments per load.  (G is even or there is one row.)
    constexpr int LOADS = kGridMaxBlocks / 64;
    auto sum_rows = [&](const unsigned short* from, unsigned int* all, unsigned int* before) {
      constexpr int BATCH = 3;  // whose loads are in flight
      for (unsigned int r0 = warp; r0 < rows; r0 += BATCH * NW) {
        unsigned int w[BATCH][LOADS];
#pragma unroll
        for (int r = 0; r < BATCH; ++r)
#pragma unroll
          for (int j = 0; j < LOADS; ++j) {
            const unsigned int row = r0 + r * NW, b = j * 64 + lane * 2, seg = row * G + b;
            w[r][j] = row < rows && b < G && seg < segs ? __ldcg(reinterpret_cast<const unsigned int*>(from + seg)) : 0u;
            if (b + 1 >= G || seg + 1 >= segs) w[r][j] &= 0xFFFFu;
          }
#pragma unroll
        for (int r = 0; r < BATCH; ++r) {
          const unsigned int row = r0 + r * NW;
          unsigned int a = 0, e = 0;
#pragma unroll
          for (int j = 0; j < LOADS; ++j) {  // (at most LOADS * 8192 in either half)
            const unsigned int b = j * 64 + lane * 2;
            a += w[r][j];
            e += b + 1 < blk ? w[r][j] : b < blk ? w[r][j] & 0xFFFFu : 0u;
          }
          a = __reduce_add_sync(FULL, (a & 0xFFFFu) + (a >> 16));
          e = __reduce_add_sync(FULL, (e & 0xFFFFu) + (e >> 16));
          if (lane == 0 && row < rows) {
            all[row] = a;
            before[row] = e;
          }
        }
      }
    };
    sum_rows(seg_s, row_s, part_s);
    if (single) sum_rows(seg_t, row_t, part_t);
  }
  uint32_t T = wlo;
  unsigned int last_idx = 0;  // keys equal to T survive up to this index
  if (!single) {
    // The rem-th largest of the bin's keys, bit by bit, then the last survivor's index if more keys equal it than survive.
    const bool both = in_bin > (unsigned)THREADS;
    auto count = [&](auto&& f) {
      unsigned int c = __syncthreads_count((unsigned)t < in_bin && f(member[0]));
      if (both) c += __syncthreads_count(t + THREADS < in_bin && f(member[1]));
      return c;
    };
    uint32_t rel = 0;
    for (uint32_t bit = 1u << (31 - __clz(max(whi - wlo - 1, 1u))); bit != 0; bit >>= 1)
      if (count([&](const uint2& m) { return m.x - wlo >= (rel | bit); }) >= rem) rel |= bit;
    T = wlo + rel;
    const unsigned int ties = rem - count([&](const uint2& m) { return m.x > T; });
    last_idx = n - 1;
    if (count([&](const uint2& m) { return m.x == T; }) != ties) {
      unsigned int less = 0;  // the largest index that fewer than `ties` of them lie below
      for (unsigned int bit = 1u << 30; bit != 0; bit >>= 1)
        if (count([&](const uint2& m) { return m.x == T && m.y < (less | bit); }) < ties) less |= bit;
      last_idx = less;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint2 m = member[u];
      if (t + u * THREADS >= in_bin || !(m.x > T || (m.x == T && m.y <= last_idx))) continue;
      const unsigned int seg = m.y / SEG, first = seg < blk ? 0u : (seg - blk) / G + 1;  // the block's first row behind it
      if (first < rows) atomicAdd(extra + first, 1u);
      if (seg < segs && seg % G == blk) {
        const unsigned int at = seg / G * PITCH, w = m.y % SEG / SLICE;
        atomicAdd(cnt + at + w, 1u);
        for (unsigned int higher = w + 1; higher < (unsigned)NW; ++higher) atomicAdd(base + at + higher, 1u);
      }
    }
  }
  __syncthreads();
  {
    // Every warp for itself, a lane per row: survivors before the segment (row_at) and of lower warps in it.
    auto scan = [&](unsigned int v) {
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned int up = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += up;
      }
      return v;
    };
    unsigned int rows_s = 0, rows_t = 0, more = 0;  // up to the 32 rows
    unsigned int cut_row = FULL, cut_rank = 0;                   // the slice that holds the last tie kept, and its rank in it
    for (unsigned int r0 = 0; r0 < rows; r0 += 32) {
      const unsigned int row = r0 + lane;
      const bool in = row < rows;
      const unsigned int all_s = in ? row_s[row] : 0u, c = in ? cnt[row * PITCH + warp] : 0u;
      const unsigned int left = in ? base[row * PITCH + warp] : 0u;  // of lower warps in the segment
      const unsigned int i_s = scan(all_s), i_x = scan(in ? extra[row] : 0u);
      unsigned int at = rows_s + i_s - all_s + (in ? part_s[row] : 0u) + more + i_x, mine = c & 0xFFFFu, before = at + (left & 0xFFFFu);
      rows_s += __shfl_sync(FULL, i_s, 31);
      more += __shfl_sync(FULL, i_x, 31);
      if (single) {  // of the ties the first `rem`
        const unsigned int all_t = in ? row_t[row] : 0u, i_t = scan(all_t), ct = c >> 16;
        const unsigned int at_t = rows_t + i_t - all_t + (in ? part_t[row] : 0u), before_t = at_t + (left >> 16);
        rows_t += __shfl_sync(FULL, i_t, 31);
        at += min(at_t, rem);
        before += min(before_t, rem);
        mine += before_t >= rem ? 0u : min(ct, rem - before_t);
        const unsigned int kept = __ballot_sync(FULL, in && ct != 0 && before_t < rem);  // (the first rows)
        if (kept != 0) {
          const int r = 31 - __clz(kept);
          last_idx = min(row_index(r0 + r) + SLICE, n) - 1;
          const unsigned int rank = rem - __shfl_sync(FULL, before_t, r);
          cut_row = rank < __shfl_sync(FULL, ct, r) ? r0 + r : FULL;
          cut_rank = rank;
        }
      }
      if (in) {
        base[row * PITCH + warp] = before;
        cnt[row * PITCH + warp] = mine;
        row_at[row] = at;  // (every warp the same)
      }
    }
    if (blk == 0 && t == 0 && rows_s + (single ? min(rows_t, rem) : rem) != k) set_status(&p.ctl->status, NSML_ERR_INTERNAL);
    __syncwarp();
    if (cut_row != FULL) {  // (one warp of the grid)
      unsigned int seen = 0;
      if (len > cap || T == 0) {  // (zeros may not be listed)
        walk_slices([&](unsigned int row) { return row == cut_row; }, [&](unsigned int row, const uint32_t (&bits)[EPL], int here, unsigned int) {
          unsigned int mine = 0, all, at = FULL;
#pragma unroll
          for (int e = 0; e < EPL; ++e) mine += (bits[e] & 0x7FFFFFFFu) == T && e < here;
          unsigned int rank = lanes_before(mine, all);
#pragma unroll
          for (int e = 0; e < EPL; ++e)
            if ((bits[e] & 0x7FFFFFFFu) == T && e < here && ++rank == cut_rank) at = row_index(row) + lane * EPL + e;
          last_idx = __reduce_min_sync(FULL, at);
        });
      } else {
        walk_list([&](bool live, unsigned int row, uint32_t key, unsigned int off) {
          const bool tie = live && row == cut_row && key == T;
          const unsigned int who = __ballot_sync(FULL, tie);
          const unsigned int it = __ballot_sync(FULL, tie && seen + __popc(who & lt) == cut_rank - 1);
          if (it != 0) last_idx = row_index(cut_row) + __shfl_sync(FULL, off, __ffs(it) - 1);
          seen += __popc(who);
        });
      }
    }
  }

  // the survivors among a lane's elements
  auto survivors_of = [&](const uint32_t (&bits)[EPL], unsigned int idx) {
    unsigned int flags = 0;
    bool tie = false;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
      flags |= (unsigned)((bits[e] & 0x7FFFFFFFu) > T) << e;
      tie |= (bits[e] & 0x7FFFFFFFu) == T;
    }
    if (tie) {
#pragma unroll
      for (int e = 0; e < EPL; ++e) flags |= (unsigned)((bits[e] & 0x7FFFFFFFu) == T && idx + e <= last_idx) << e;
    }
    return flags;
  };
  auto with_survivors = [&](unsigned int row) { return cnt[row * PITCH + warp] != 0; };
  if (blk == 0 && t == 0) write_header(p);
  uint32_t* out_idx = reinterpret_cast<uint32_t*>(p.payload + p.P.idx_off);
  const bool int8 = p.bits == NSML_BITS_INT8;
  signed char* out8 = reinterpret_cast<signed char*>(p.payload + p.P.val_off);
  // The offsets of a slice's survivors are put in order, then index and value are written 32 at a time.  (Every lane writing
  // its own survivors, four or eight stores that each touch ten to twenty sectors: 48 us for 64M bfloat16 at 0.1, so 24.)
  auto write_slices = [&](auto&& value) {  // value(scale, place, bits, index)
    walk_slices(with_survivors, [&](unsigned int row, const uint32_t (&bits)[EPL], int, unsigned int kept_at) {
      const unsigned int i0 = row_index(row), flags = survivors_of(bits, i0 + lane * EPL), first = base[row * PITCH + warp];
      unsigned int all, rank = lanes_before(__popc(flags), all);
#pragma unroll
      for (int e = 0; e < EPL; ++e)
        if (flags & (1u << e)) sh.stage[warp][rank++] = (unsigned char)(lane * EPL + e);
      const void* from = s_slice + (kept_at - 1) * 32;
      if (kept_at == kNotHere) {
        sh.slice[warp][lane] = pack(bits);
        from = sh.slice[warp];
      }
      __syncwarp();
      if (first + all <= k) {
        SliceScale scale = {0.f, 0.f, row * SLOTS - row_at[row] / NSML_QBLOCK, first / NSML_QBLOCK == (first + all - 1) / NSML_QBLOCK};
        scale.scale = __uint_as_float(qm[scale.slots + first / NSML_QBLOCK]);  // (int8)
        scale.inv = __uint_as_float(qi[scale.slots + first / NSML_QBLOCK]);
        uint32_t* to = out_idx + first;
#pragma unroll 2
        for (unsigned int j = lane; j < all; j += 32) {
          const unsigned int off = sh.stage[warp][j], idx = i0 + off;
          const uint32_t b = PACKED ? (uint32_t)static_cast<const unsigned short*>(from)[off] << 16 : static_cast<const uint32_t*>(from)[off];
          to[j] = idx;
          value(scale, first + j, b, idx);
        }
      }
      __syncwarp();
    });
  };
  if (p.bits == NSML_BITS_FP16) {
    uint16_t* out16 = reinterpret_cast<uint16_t*>(p.payload + p.P.val_off);
    write_slices([&](const SliceScale&, unsigned int at, uint32_t bits, unsigned int idx) {
      const uint16_t h = encode_f16(__uint_as_float(bits));
      out16[at] = h;
      if (FEEDBACK && bits != 0) residual[idx] = __fsub_rn(__uint_as_float(bits), decode_f16(h));  // (+0.0: see not_carried)
    });
    return;
  }
  if (!int8) {
    write_slices([&](const SliceScale&, unsigned int at, uint32_t bits, unsigned int idx) {
      put_value(p, at, bits);
      if (FEEDBACK && bits != 0) residual[idx] = not_carried(p, bits);  // (+0.0: see not_carried)
    });
    return;
  }
  // int8: the largest magnitude of every payload block.  A slice's largest key is a survivor if it has any: a lane per slice,
  // but where a slice's survivors lie in two payload blocks.
  for (unsigned int r0 = 0; r0 < rows; r0 += 32) {
    const unsigned int row = r0 + lane, mine = row < rows ? cnt[row * PITCH + warp] : 0u;
    if (mine != 0) {
      const unsigned int first = base[row * PITCH + warp], last = first + mine - 1;
      if (first / NSML_QBLOCK == last / NSML_QBLOCK && last < k)
        atomicMax(qm + (row * SLOTS + first / NSML_QBLOCK - row_at[row] / NSML_QBLOCK), top[row * PITCH + warp]);
    }
  }
  walk_slices([&](unsigned int row) {
    const unsigned int first = base[row * PITCH + warp], mine = cnt[row * PITCH + warp];
    return mine != 0 && first / NSML_QBLOCK != (first + mine - 1) / NSML_QBLOCK && first + mine <= k;
  }, [&](unsigned int row, const uint32_t (&bits)[EPL], int, unsigned int) {
    const unsigned int flags = survivors_of(bits, row_index(row) + lane * EPL), slots = row * SLOTS - row_at[row] / NSML_QBLOCK;
    unsigned int all, at = base[row * PITCH + warp] + lanes_before(__popc(flags), all);
#pragma unroll
    for (int e = 0; e < EPL; ++e)
      if (flags & (1u << e)) atomicMax(qm + (slots + at++ / NSML_QBLOCK), bits[e] & 0x7FFFFFFFu);  // (slots may be below zero)
  });
  __syncthreads();
  for (unsigned int i = t; i < rows * SLOTS; i += THREADS)
    if (qm[i]) atomicMax(qmax + row_at[i / SLOTS] / NSML_QBLOCK + i % SLOTS, qm[i]);
  if (!grid_barrier(p.ctl, ++barriers * G, sh)) return;

  // ---------------- int8: scales and codes ----------------
  for (unsigned long long i = (unsigned long long)blk * THREADS + t; i < p.P.nblocks; i += (unsigned long long)G * THREADS)
    reinterpret_cast<float*>(p.payload + p.P.scale_off)[i] = __fdiv_rn(__uint_as_float(__ldcg(qmax + i)), 127.0f);
  for (unsigned int i = t; i < rows * SLOTS; i += THREADS)
    if (qm[i]) {  // (0: nothing but zeros there, whose code is 0 whatever the scale)
      const float scale = __fdiv_rn(__uint_as_float(__ldcg(qmax + row_at[i / SLOTS] / NSML_QBLOCK + i % SLOTS)), 127.0f);
      qm[i] = __float_as_uint(scale);
      qi[i] = __float_as_uint(__fdiv_rn(1.0f, scale));
    }
  __syncthreads();
  write_slices([&](const SliceScale& c, unsigned int at, uint32_t bits, unsigned int idx) {
      float scale = c.scale, inv = c.inv;
      if (!c.one) {
        scale = __uint_as_float(qm[c.slots + at / NSML_QBLOCK]);
        inv = __uint_as_float(qi[c.slots + at / NSML_QBLOCK]);
      }
      const float v = __uint_as_float(bits);
      const int code = encode_i8(v, scale, inv);
      out8[at] = (signed char)code;
      if (FEEDBACK && v != 0.0f) residual[idx] = __fsub_rn(v, decode_i8(code, scale));  // (a zero: as in quantize_group)
    });
}

template <int DTYPE>
using GridKernel = void (*)(BucketSrc<DTYPE>, FinalizeParams, unsigned int, unsigned int, unsigned int, unsigned int, unsigned int, unsigned int);
// The instances for large buckets are compiled beside the others, in nsml_grid_large.cu.
template <int DTYPE>
GridKernel<DTYPE> large_grid_kernel(bool feedback, bool masked);

}  // namespace nsml
