// Decompress and sum the W gathered payloads into one dense float32 gradient
// (Section 4.2 Step 3 "further aggregation"; with top-k payloads every worker
// receives all payloads, the AllGather pattern of Section 5.3, and sums them).
//
// Payload indices are ascending, so the work is split by dense range instead
// of by payload entry: a block owns a tile of the dense buffer, finds each
// worker's entries for that tile from a precomputed offset table, adds them in
// worker order in shared memory and writes the tile once, coalesced.  No
// atomics, fixed summation order, and in overwrite mode the zero fill costs
// nothing extra.
#pragma once

#include "nsml_common.cuh"
#include "nsml_codec.cuh"

namespace nsml {

// Dense elements per tile (the block's unit of work; 32 or 8 KB of shared memory).  The small tile spreads a short
// bucket's entries, and the round trips they take, over more blocks; it is taken while its blocks are one wave (1024
// tiles; 7 blocks on each of 148 SMs are 1036), with a margin of a few.  Measured (us per sum, several in a row, small /
// large tile).  Overwriting, W = 4 at 0.01 int8: 300k elements 7.9 / 8.4, 1M 10.0 / 9.9, 2.0M 11.9 / 11.5, 2.4M (a second
// wave) 14.5 / 11.9; W = 2 at 0.3 float32: 1M 14.3 / 17.7, 2.0M 18.2 / 20.6.  Adding, W = 4 at 0.01: 300k 8.8 / 11.6, 1M
// 12.4 / 18.1, 2.0M 14.6 / 20.0, 2.4M 19.5 / 20.1.  The large one's lead where a bucket of 1 to 2M elements is
// overwritten with few entries is 7 per cent at most, the small one's where it is added to 30.
constexpr int kDenseTileLarge = 8192;
constexpr int kDenseTileSmall = 2048;
constexpr int64_t kDenseTileSmallMaxN = 1024LL * kDenseTileSmall;
static_assert(kDenseTileLarge == 1 << 13 && kDenseTileSmall == 1 << 11, "tiles by shift");
inline int dense_tile(int64_t n) { return n <= kDenseTileSmallMaxN ? kDenseTileSmall : kDenseTileLarge; }

struct PayloadTable {
  const unsigned char* p[NSML_MAX_WORKERS];
  unsigned long long bytes[NSML_MAX_WORKERS];  // size of the buffer behind p[w]; 0 = not known
};

struct AccumulateLayout {
  size_t offsets;  // u32[W][tiles + 1]
  size_t total;    // what a sum of n elements uses
  size_t ask;      // what a caller is told to bring: enough for every smaller n, too (one workspace serves buckets of
                   // several sizes), although the table is shorter right above kDenseTileSmallMaxN than below it
};

inline AccumulateLayout accumulate_layout(int64_t n, int W) {
  AccumulateLayout L;
  const size_t tile = (size_t)dense_tile(n), tiles = ((size_t)n + tile - 1) / tile;
  const size_t most_small = ((size_t)kDenseTileSmallMaxN + kDenseTileSmall - 1) / kDenseTileSmall;
  L.offsets = 256;
  L.total = L.offsets + align_up((size_t)W * (tiles + 1) * 4, 256);
  L.ask = n <= kDenseTileSmallMaxN || tiles >= most_small ? L.total : L.offsets + align_up((size_t)W * (most_small + 1) * 4, 256);
  return L;
}

// A header is accepted when its fields describe a payload for this n in the layout nsml_compress writes
// and, where the size of the buffer is known (bytes != 0), that layout fits the buffer: a truncated
// payload, or one whose k field was corrupted upwards, is then refused before anything behind the header
// is read.
__host__ __device__ inline bool header_ok(const nsml_payload_header* h, unsigned long long n, unsigned long long bytes = 0) {
  if (h->magic != NSML_PAYLOAD_MAGIC || h->version != NSML_PAYLOAD_VERSION) return false;
  if (h->n != n || h->k < 1 || h->k > n || h->qblock != NSML_QBLOCK) return false;
  if (h->bits != NSML_BITS_INT8 && h->bits != NSML_BITS_FP16 && h->bits != NSML_BITS_FP32) return false;
  const unsigned long long k = h->k;
  const unsigned long long val_off = 64 + (k * 4 + 15) / 16 * 16;
  if (h->idx_off != 64 || h->val_off != val_off) return false;
  unsigned long long total;
  if (h->bits == NSML_BITS_INT8) {
    const unsigned long long nblocks = (k + NSML_QBLOCK - 1) / NSML_QBLOCK;
    if (h->nblocks != nblocks) return false;
    if (h->scale_off != val_off + (k + 15) / 16 * 16) return false;
    total = h->scale_off + (nblocks * 4 + 15) / 16 * 16;
  } else {
    total = val_off + (k * (h->bits == NSML_BITS_FP32 ? 4 : 2) + 15) / 16 * 16;
  }
  return bytes == 0 || total <= bytes;
}

// offsets[w][b] = first payload entry of worker w whose index is >= b * tile.
//
// What bounds the kernel is its chain of dependent reads (about 1 us each from DRAM).  Payloads of few entries are read
// as a whole (kPartScan, kPartShare): a thread compares the tiles of four neighbouring entries and writes the boundaries between
// them, so that there are two reads in a row, header and indices; and the indices are in L2 when the sum reads them.
// Where that is more to read than a search (every entry against some 200 bytes per boundary), a block settles
// kPartBounds consecutive boundaries of one worker, a thread each: kPartProbes evenly spaced indices of the whole array go
// to shared memory (and, where the block's boundaries lie in a small part of it, as many of that part: about one
// probe per boundary); every thread finds the two probes around its boundary there, interpolates between them and
// counts in the 16 entries around the guess, which settles the boundary in one read wherever the indices are
// locally even, and gallops from the guess where they are not: three or four dependent reads with the payload
// header's.  (350M elements, 8 workers, 342k boundaries: 54 us with a binary search per thread, 43 us now;
// 25M elements, 4 workers of 250k entries: 12.3 us with a binary search, 10.4 with the probes, 6 read as a whole; 1M, 2
// workers of 52k: 6.2 with the probes, 3.5.  The launch may start under the kernel before it.  Sum as a whole: 25M 35.2 ->
// 29.1 us, 1M added to 12.3 -> 9.6.)
//
// The sum's kernel may be launched once the blocks with nothing to do have left: placed around them (16 of 17 where the
// payloads turn out to be searched, each holding half an SM's registers) its blocks are spread unevenly.  Eight payloads of
// 655k entries, searched, in 6.55M elements: 63.8 -> 59.2 us, of 10M in 25M 229.8 -> 221; read as a whole, 250k in 25M: 29.2 ->
// 28.5.
//
// The kernel also clears the call's status word (no separate clearing step is needed); payload errors are
// reported by the merge kernel: a worker with a bad header gets all-zero offsets, so nothing of its payload
// is read.  In a corrupt payload, whose indices do not ascend or lie beyond the last tile, boundaries may be written more
// than once, by any of several entries, but each is written: on the way from before the first tile to behind the last one
// the indices pass it upwards.  Boundary 0 is 0, so if the last one is the number of entries, the ranges of the tiles cover
// every entry, in whichever order they run, and an entry in a range that is not its tile's is found by the merge kernel,
// which also takes no offset beyond the number of entries.
constexpr int kPartBounds = 1024;
constexpr unsigned int kPartProbes = kPartBounds;  // one per thread
constexpr unsigned int kPartWindow = 16;
constexpr unsigned int kPartScan = 8u << 20;  // entries of all workers up to which they are read as a whole: 32 MB, 5 us (the
                                              // line below is lower, but for 8 workers from 537M elements on, 64 from 67M)
constexpr unsigned int kPartParts = 64;       // blocks per worker for that, at most
constexpr unsigned int kPartShare = 16384;    // ... and entries per block: four rounds of its threads
// Blocks per worker: 8192 entries each of the largest payload, as far as the buffers' sizes tell (an entry takes five bytes
// at least), otherwise of an 8th of the bucket.  At most 128 for all workers, because blocks that find little to do still hold half an
// SM each until the kernel before them is done and the header is there: 64 for each of eight workers made four streams' steps
// 20 % longer and sums of eight dense payloads 5 %.  (many_calls: nsml_set_list_block_candidates above its default.)
inline unsigned int partition_blocks(int64_t n, unsigned int tiles, int W, unsigned long long largest_payload, bool many_calls) {
  const unsigned int search = tiles / kPartBounds + 1;
  const unsigned long long entries = largest_payload != 0 ? largest_payload / 5 : (unsigned long long)n / 8;
  unsigned int most = 128u / W;
  if (most < 1) most = 1;
  if (most > kPartParts) most = kPartParts;
  if (many_calls) most = (most + 3) / 4;
  const unsigned long long scan = entries / 8192 + 1;
  const unsigned int parts = scan < most ? (unsigned int)scan : most;
  return search > parts ? search : parts;
}

// [lo, hi] of the first entry whose index is >= target: entries below lo are below it, entry hi is not (or hi is
// the end).  The probes in shared memory are every gap-th entry from `base` on, `count` of them.
__device__ __forceinline__ unsigned int probe_bracket(const uint32_t* s_probe, unsigned int count, unsigned int base, unsigned int gap,
                                                      unsigned int end, unsigned int target, unsigned int& lo, unsigned int& hi) {
  unsigned int a = 0, b = count;  // first probe that is >= target
  while (a < b) {
    const unsigned int mid = (a + b) >> 1;
    if (s_probe[mid] < target) a = mid + 1; else b = mid;
  }
  lo = a == 0 ? base : base + (a - 1) * gap + 1;
  hi = a == count ? end : base + a * gap;
  return a;
}

// Writes `value` for boundaries b .. last, by a warp.
__device__ __forceinline__ void fill_bounds(unsigned int* out, unsigned int b, unsigned int last, unsigned int value) {
  for (b += threadIdx.x & 31; b <= last; b += 32) out[b] = value;
}

// Boundaries of a payload that is read as a whole; part: the block's of `parts`.
__device__ __forceinline__ void scan_bounds(const uint32_t* idx, unsigned int k, unsigned int tiles, unsigned int shift, unsigned int part,
                                            unsigned int parts, unsigned int* out) {
  constexpr unsigned int FULL = 0xFFFFFFFFu;
  const unsigned int lane = threadIdx.x & 31, quads = (k + 3) / 4, per = (quads + parts - 1) / parts;
  const unsigned int begin = part * per, end = min(quads, begin + per);
  for (unsigned int q0 = begin + (threadIdx.x & ~31u); q0 < end; q0 += kPartBounds) {  // uniform over the warp
    const unsigned int q = q0 + lane;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (q < end) v = __ldg(reinterpret_cast<const uint4*>(idx) + q);  // (the section is padded)
    unsigned int before = __shfl_up_sync(FULL, v.w, 1);
    if (lane == 0 && q0 != 0) before = __ldg(idx + 4ull * q0 - 1);
    const uint32_t e[4] = {v.x, v.y, v.z, v.w};
    unsigned int next = q == 0 ? 0u : min(before >> shift, tiles) + 1;  // the first boundary behind the entry before
#pragma unroll
    for (unsigned int i = 0; i < 4; ++i) {
      const unsigned int j = 4 * q + i, reach = q < end && j < k ? min(e[i] >> shift, tiles) + 1 : next;  // boundaries next .. reach - 1 are the entry's
      const bool many = reach > next + 4;
      if (!many)
        for (unsigned int b = next; b < reach; ++b) out[b] = j;
      for (unsigned int left = __ballot_sync(FULL, many); left != 0; left &= left - 1) {
        const int who = __ffs(left) - 1;
        fill_bounds(out, __shfl_sync(FULL, next, who), __shfl_sync(FULL, reach, who) - 1, __shfl_sync(FULL, j, who));
      }
      if (q < end && j < k) next = reach;
    }
    const unsigned int last = __ballot_sync(FULL, q < end && q == quads - 1);  // behind the last entry
    if (last != 0) fill_bounds(out, __shfl_sync(FULL, next, __ffs(last) - 1), tiles, k);
  }
}

__global__ void __launch_bounds__(kPartBounds)
k_partition(PayloadTable table, int W, unsigned long long n, unsigned int tiles, unsigned int tile_shift,
            unsigned int* __restrict__ offsets, int* status) {
  __shared__ uint32_t s_probe[kPartProbes];
  pdl_wait();
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *status = NSML_OK;
  const int w = blockIdx.y;
  const unsigned int first = blockIdx.x * kPartBounds, count = first > tiles ? 0u : min((unsigned)kPartBounds, tiles + 1 - first);
  const unsigned int tile_elems = 1u << tile_shift;
  unsigned int* all = offsets + (unsigned long long)w * (tiles + 1ull);
  unsigned int* out = all + first;
  const nsml_payload_header* h = reinterpret_cast<const nsml_payload_header*>(table.p[w]);
  if (!header_ok(h, n, table.bytes[w])) {  // uniform over the block
    if (threadIdx.x < count) out[threadIdx.x] = 0;
    return;
  }
  const uint32_t* idx = reinterpret_cast<const uint32_t*>(table.p[w] + h->idx_off);
  const unsigned int parts = min(gridDim.x, kPartParts);
  if (h->k * (unsigned long long)W <= kPartScan && h->k <= parts * (unsigned long long)kPartShare) {
    if (blockIdx.x >= parts) return;
    pdl_launch_dependents();
    scan_bounds(idx, (unsigned int)h->k, tiles, tile_shift, blockIdx.x, parts, all);
    return;
  }
  if (count == 0) return;
  pdl_launch_dependents();
  unsigned int base = 0, end = (unsigned int)h->k;  // k <= n < 2^31; so is every target below: (tiles + 1) * tile < 2^32
  unsigned int gap, probes, from, to, a;
  auto probe = [&]() {
    gap = (end - base + kPartProbes - 1) / kPartProbes;
    probes = gap == 0 ? 0u : (end - base + gap - 1) / gap;
    if (threadIdx.x < probes) s_probe[threadIdx.x] = __ldg(idx + base + threadIdx.x * gap);
    __syncthreads();
  };
  probe();
  unsigned int lo, hi, unused;
  probe_bracket(s_probe, probes, base, gap, end, first * tile_elems, lo, unused);
  probe_bracket(s_probe, probes, base, gap, end, (first + count - 1) * tile_elems, unused, hi);
  if (gap > kPartWindow && (unsigned long long)(hi - lo) * 4 < end - base) {  // (hi < lo, in a corrupt payload only, fails this)
    base = lo;
    end = hi;
    __syncthreads();  // the probes have been read
    probe();
  }
  if (threadIdx.x >= count) return;
  const unsigned int target = (first + threadIdx.x) * tile_elems;
  a = probe_bracket(s_probe, probes, base, gap, end, target, from, to);
  unsigned int guess = from + (to - from) / 2;
  if (a != 0 && a != probes && from < to) {
    const unsigned int below = s_probe[a - 1], reach = s_probe[a];
    if (below < target && target <= reach) guess = from + min((unsigned int)((float)(to - from) * ((float)(target - below) / (float)(reach - below))), to - from);
  }
  unsigned int stride = kPartWindow;
  while (from < to) {
    const unsigned int start = max((int)guess - (int)kPartWindow / 2, (int)from) & ~3u;  // 16-byte aligned; the section is padded
    uint4 v[kPartWindow / 4];
#pragma unroll
    for (unsigned int i = 0; i < kPartWindow / 4; ++i)
      v[i] = start + i * 4 < to ? __ldg(reinterpret_cast<const uint4*>(idx + start) + i) : make_uint4(0u, 0u, 0u, 0u);
    unsigned int seen = 0, less = 0;
#pragma unroll
    for (unsigned int i = 0; i < kPartWindow / 4; ++i) {
      const uint32_t e[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
#pragma unroll
      for (unsigned int q = 0; q < 4; ++q) {
        const unsigned int j = start + i * 4 + q;
        seen += j >= from && j < to;
        less += j >= from && j < to && e[q] < target;
      }
    }
    const unsigned int first_seen = max(start, from);
    if (less == 0) {
      to = first_seen;
      guess = to - min(stride, (to - from) / 2);
    } else if (less == seen) {
      from = first_seen + seen;
      guess = from + min(stride, (to - from) / 2);
    } else {
      from = to = first_seen + less;
    }
    stride *= 4;
  }
  out[threadIdx.x] = from;
}

// What a block needs to know about one worker's payload, read from its header once per block.
struct WorkerView {
  const uint32_t* idx;
  const unsigned char* val;  // int8 codes, binary16 bit patterns or float32 values
  const float* scale;
  int bits;
};

constexpr int kMergeThreads = 128;
constexpr int kMergeUnits = 4;  // units whose loads are in flight before the first one's adds are applied

// Four consecutive payload entries: as loaded, and decoded to (slot of the tile, value).
struct MergeQuad {
  uint4 idx, val;  // val: 4, 8 or 16 bytes of it used
  float scale;
  int first, last;  // entries first .. last-1 of the four count (nothing of what was loaded is touched before the
                    // adds, so that the loads of several quads are in flight together)

  // entries j .. j+3 (j a multiple of 4; the sections are padded to 16 bytes) of those in [from, to)
  __device__ __forceinline__ void load(const WorkerView& v, unsigned int j, unsigned int from, unsigned int to) {
    first = max(0, (int)from - (int)j);
    last = min(4, (int)to - (int)j);
    if (last <= 0) return;
    idx = __ldcs(reinterpret_cast<const uint4*>(v.idx + j));
    if (v.bits == NSML_BITS_INT8) {
      val.x = __ldcs(reinterpret_cast<const unsigned int*>(v.val + j));
      scale = __ldg(v.scale + (j >> 10));
    } else if (v.bits == NSML_BITS_FP16) {
      const uint2 t = __ldcs(reinterpret_cast<const uint2*>(v.val + 2ull * j));
      val.x = t.x; val.y = t.y;
    } else {
      val = __ldcs(reinterpret_cast<const uint4*>(v.val + 4ull * j));
    }
  }

  __device__ __forceinline__ void values(int bits, float (&v)[4]) const {
    if (bits == NSML_BITS_INT8) {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = decode_i8((int)(signed char)(val.x >> (8 * e)), scale);
    } else if (bits == NSML_BITS_FP16) {
      v[0] = decode_f16((uint16_t)val.x); v[1] = decode_f16((uint16_t)(val.x >> 16));
      v[2] = decode_f16((uint16_t)val.y); v[3] = decode_f16((uint16_t)(val.y >> 16));
    } else {
      v[0] = __uint_as_float(val.x); v[1] = __uint_as_float(val.y);
      v[2] = __uint_as_float(val.z); v[3] = __uint_as_float(val.w);
    }
  }
};

// Persistent blocks, tile-cyclic.  A tile's entries are taken worker by worker in units of 128 aligned quads (four
// consecutive entries), a quad per thread: one 16-byte load fetches four indices, and everything but the quad's own
// data is uniform over the block.  The loads of kMergeUnits units are issued together, then the units' adds are
// applied in order, with a block barrier wherever the worker changes: an element gets at most one add per worker,
// in worker order.  A full tile leaves by one bulk copy from shared memory.
//
// Measured (one B200).  Eight payloads of 17.5M entries into 350M elements, 2.1 GB: 732 us when a thread took one
// entry per unit (about 130 instructions per entry and thread: issue-bound), about 425 us now (4.9 TB/s); four
// payloads of 250k entries into 25M elements, 105 MB: 29.9 -> 25.5 us, of which 19.8 us are the writes alone.
// Two things made the difference beside the quads: everything but the data is uniform over the block (a flat list
// of quads over all workers, with a search for the quad's worker, took 743 us), and nothing that was loaded is
// touched before the adds (masking the edge entries in the loaded registers made every unit wait for its own loads:
// 671 us).
template <int TILE>
__global__ void __launch_bounds__(kMergeThreads, 7)
k_merge(PayloadTable table, int W, float* __restrict__ dense, unsigned long long n, int zero_first,
        unsigned int tiles, const unsigned int* __restrict__ offsets, int* status) {
  __shared__ __align__(128) float s_acc[TILE + 1];  // the last slot takes the adds of entries that do not exist
  __shared__ WorkerView s_view[NSML_MAX_WORKERS];
  __shared__ uint2 s_range[2][NSML_MAX_WORKERS];  // the tile's entries of every worker; double-buffered
  const unsigned long long per = (unsigned long long)tiles + 1;
  bool bad = false;
  unsigned int entries = 0;  // of worker threadIdx.x
  if (threadIdx.x < W) {
    // Headers are checked here (the partition kernel cleared the status word).  A worker with a bad
    // header has all-zero offsets, so its view is never used.
    const unsigned char* pbase = table.p[threadIdx.x];
    const nsml_payload_header* h = reinterpret_cast<const nsml_payload_header*>(pbase);
    WorkerView v = {nullptr, nullptr, nullptr, 0};
    if (header_ok(h, n, table.bytes[threadIdx.x])) {
      v.idx = reinterpret_cast<const uint32_t*>(pbase + h->idx_off);
      v.val = pbase + h->val_off;
      v.scale = reinterpret_cast<const float*>(pbase + h->scale_off);
      v.bits = (int)h->bits;
      entries = (unsigned int)h->k;
    } else {
      bad = blockIdx.x == 0;
    }
    s_view[threadIdx.x] = v;
  }
  pdl_wait();  // the offsets are complete
  const unsigned int* my_offsets = offsets + threadIdx.x * per;  // thread w looks after worker w's ranges
  if (threadIdx.x < W && blockIdx.x == 0) bad |= __ldcg(my_offsets + tiles) != entries;  // (there are entries behind the last tile)
  if (threadIdx.x < W && blockIdx.x < tiles) s_range[0][threadIdx.x] = make_uint2(min(entries, __ldcg(my_offsets + blockIdx.x)), min(entries, __ldcg(my_offsets + blockIdx.x + 1)));
  int buf = 0;
  for (unsigned int tile = blockIdx.x; tile < tiles; tile += gridDim.x, buf ^= 1) {
    const unsigned long long lo = (unsigned long long)tile * TILE;
    const unsigned int len = (unsigned int)min((unsigned long long)TILE, n - lo);
    float* dtile = dense + lo;
    if (threadIdx.x == 0) bulk_store_wait_read();  // the previous tile has left shared memory
    __syncthreads();  // this tile's ranges (first tile: the views too) are in place
    const uint2* range = s_range[buf];
    // the next tile's ranges are fetched while this tile is summed
    uint2 ahead = make_uint2(0u, 0u);
    const bool fetch = threadIdx.x < W && (unsigned long long)tile + gridDim.x < tiles;
    if (fetch) ahead = make_uint2(__ldcg(my_offsets + tile + gridDim.x), __ldcg(my_offsets + tile + gridDim.x + 1));

    bool staged = zero_first;
    if (!zero_first) {
      // Adding few entries to what dense holds: touch only their elements in global memory.  Otherwise the tile
      // is staged in shared memory and written in one sweep.
      unsigned int total = 0;
      for (int w = 0; w < W; ++w) total += max(range[w].y, range[w].x) - range[w].x;
      staged = total * 64ull > len;
    }
    if (zero_first) {
#pragma unroll
      for (unsigned int i = 0; i < TILE; i += kMergeThreads * 4)
        *reinterpret_cast<float4*>(s_acc + i + threadIdx.x * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
    } else if (staged) {
      for (unsigned int i = threadIdx.x * 4; i < len; i += kMergeThreads * 4) {
        if (i + 4 <= len) *reinterpret_cast<float4*>(s_acc + i) = *reinterpret_cast<const float4*>(dtile + i);
        else for (unsigned int e = i; e < len; ++e) s_acc[e] = dtile[e];
      }
    }
    // (w, c): the next unit is quads c .. c+127 of worker w's; uniform over the block.  A range that runs
    // backwards (a corrupt, unsorted payload) counts as empty.
    int w = 0;
    unsigned int c = 0;
    while (w < W && range[w].x >= range[w].y) ++w;
    bool placed = false;  // the tile's starting values are known to be in place
    while (w < W) {
      MergeQuad q[kMergeUnits];
      int unit_w[kMergeUnits];
      int unit_bits[kMergeUnits];
#pragma unroll
      for (int u = 0; u < kMergeUnits; ++u) {
        unit_w[u] = w;
        if (w < W) {
          const uint2 r = range[w];
          const WorkerView v = s_view[w];
          unit_bits[u] = v.bits;
          const unsigned int first = (r.x & ~3u) + c * 4;
          q[u].load(v, first + threadIdx.x * 4, r.x, r.y);
          c += kMergeThreads;
          if (first + kMergeThreads * 4 >= r.y) {  // worker w is used up: on to the next one that has entries here
            c = 0;
            do ++w; while (w < W && range[w].x >= range[w].y);
          }
        }
      }
      if (!placed) __syncthreads();
      placed = true;
#pragma unroll
      for (int u = 0; u < kMergeUnits; ++u) {
        if (unit_w[u] >= W) break;
        if (q[u].last > 0) {
          const uint32_t ix[4] = {q[u].idx.x, q[u].idx.y, q[u].idx.z, q[u].idx.w};
          float v[4];
          q[u].values(unit_bits[u], v);
          unsigned int at[4];
          bool plain = q[u].first == 0 && q[u].last == 4;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            at[e] = ix[e] - (unsigned int)lo;  // wraps if the index is below lo
            plain &= at[e] < len;
          }
          if (!plain) {  // the edges of a worker's range, or an index that does not belong here
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const bool mine = e >= q[u].first && e < q[u].last;
              bad |= mine && at[e] >= len;
              if (!mine || at[e] >= len) at[e] = TILE;
            }
          }
          if (staged) {
#pragma unroll
            for (int e = 0; e < 4; ++e) s_acc[at[e]] += v[e];
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (at[e] < TILE) dtile[at[e]] += v[e];
          }
        }
        if ((u + 1 == kMergeUnits ? w : unit_w[u + 1]) != unit_w[u]) __syncthreads();  // uniform over the block
      }
    }
    if (fetch) s_range[buf ^ 1][threadIdx.x] = make_uint2(min(entries, ahead.x), min(entries, ahead.y));
    if (!staged) continue;
    if (len == TILE) {
      fence_async_shared();
      __syncthreads();
      if (threadIdx.x == 0) bulk_store(dtile, s_acc, TILE * 4);
    } else {
      __syncthreads();
      for (unsigned int i = threadIdx.x * 4; i < len; i += kMergeThreads * 4) {
        if (i + 4 <= len) *reinterpret_cast<float4*>(dtile + i) = *reinterpret_cast<const float4*>(s_acc + i);
        else for (unsigned int e = i; e < len; ++e) dtile[e] = s_acc[e];
      }
    }
  }
  if (threadIdx.x == 0) bulk_store_wait_read();  // shared memory may not go away under a copy
  if (bad) set_status(status, NSML_ERR_PAYLOAD);
}

}  // namespace nsml
