// libnsml C ABI: argument checks, workspace carving and kernel launches.
// See include/nsml.h for the contract of every entry point.
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "nsml_accumulate.cuh"
#include "nsml_adaptive.cuh"
#include "nsml_codec.cuh"
#include "nsml_common.cuh"
#include "nsml_compact.cuh"
#include "nsml_finalize.cuh"
#include "nsml_grid.cuh"
#include "nsml_list.cuh"
#include "nsml_select.cuh"
#include "nsml_small.cuh"

namespace nsml {

// A CUDA call failed: what the call returns.  The runtime keeps the error of a refused launch or copy for the thread's next
// cudaGetLastError, which is not to meet it again: the calls that follow have nothing to do with it.  (Every launch is
// checked by its own return code.)
static int cuda_error() {
  cudaGetLastError();
  return NSML_ERR_CUDA;
}

enum KernelId {
  K_SAMPLE = 0, K_COMPACT_BUCKET, K_EMIT, K_PARTITION, K_MERGE, K_CLEAR, K_SELECT_GRID,
  K_SUMSQ, K_PRUNE_PASS, K_PRUNE_FINISH, K_SELECT_SMALL, K_COUNT
};

static const char* const kKernelNames[K_COUNT] = {"k_sample", "k_compact_bucket", "k_emit", "k_partition", "k_merge",
                                                  "k_clear", "k_select_grid", "k_sumsq", "k_prune_pass", "k_prune_finish",
                                                  "k_select_small"};

static std::atomic<int64_t> g_launches{0};

// ---- optional per-kernel timing with CUDA events --------------------------
struct ProfRecord {
  int id;
  cudaEvent_t start, stop;
};
static std::mutex g_prof_mutex;
static std::atomic<bool> g_prof_on{false};
static std::vector<ProfRecord> g_prof_records;
static double g_prof_ms[K_COUNT];
static int64_t g_prof_launches[K_COUNT];

static void prof_drain_locked() {
  for (ProfRecord& r : g_prof_records) {
    float ms = 0.f;
    if (cudaEventSynchronize(r.stop) == cudaSuccess && cudaEventElapsedTime(&ms, r.start, r.stop) == cudaSuccess) {
      g_prof_ms[r.id] += ms;
      g_prof_launches[r.id] += 1;
    }
    cudaEventDestroy(r.start);
    cudaEventDestroy(r.stop);
  }
  g_prof_records.clear();
}

struct LaunchScope {  // brackets one kernel launch
  int id;
  cudaStream_t stream;
  cudaEvent_t start = nullptr, stop = nullptr;
  // timed = false: never bracket this launch with events (creating events allocates)
  LaunchScope(int id_, cudaStream_t s, bool timed = true) : id(id_), stream(s) {
    if (timed && g_prof_on.load(std::memory_order_relaxed)) {
      cudaEventCreate(&start);
      cudaEventCreate(&stop);
      cudaEventRecord(start, stream);
    }
  }
  ~LaunchScope() {
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (start) {
      cudaEventRecord(stop, stream);
      std::lock_guard<std::mutex> lock(g_prof_mutex);
      g_prof_records.push_back({id, start, stop});
    }
  }
};

template <int DTYPE>
static GridKernel<DTYPE> grid_kernel(bool feedback, bool masked, bool large) {
  if (large) return large_grid_kernel<DTYPE>(feedback, masked);
  return feedback ? (masked ? k_select_grid<DTYPE, true, true, false> : k_select_grid<DTYPE, true, false, false>)
                  : (masked ? k_select_grid<DTYPE, false, true, false> : k_select_grid<DTYPE, false, false, false>);
}

// ---- per-device launch geometry -------------------------------------------
struct DeviceInfo {
  bool ready = false;
  int sms = 0;
  int merge_small = 0, merge_large = 0, grid = 0, sumsq = 0;  // resident blocks per SM
};
static DeviceInfo g_dev[64];
static std::mutex g_dev_mutex;

static int device_info(const DeviceInfo** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cuda_error();
  std::lock_guard<std::mutex> lock(g_dev_mutex);
  DeviceInfo& d = g_dev[dev];
  if (!d.ready) {
    if (cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return cuda_error();
    cudaError_t e = cudaSuccess;
    auto prepare = [&](auto kernel, int threads, size_t smem, int* resident) {
      if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      int r = 0;
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, kernel, threads, smem);
      if (*resident == 0 || r < *resident) *resident = r;
    };
    for (const bool feedback : {false, true})
      for (const bool masked : {false, true})
        for (const bool large : {false, true}) {
          prepare(grid_kernel<NSML_F32>(feedback, masked, large), kGridThreads, kGridSmem, &d.grid);
          prepare(grid_kernel<NSML_BF16>(feedback, masked, large), kGridThreads, kGridSmem, &d.grid);
        }
    int list_fits = 0;  // every shape of the list stage is resident at least once per SM
    prepare(k_emit<NSML_F32, kEmitPer>, kEmitThreads, sizeof(EmitShared), &list_fits);
    prepare(k_emit<NSML_BF16, kEmitPer>, kEmitThreads, sizeof(EmitShared), &list_fits);
    prepare(k_emit<NSML_F32, 2 * kEmitPer>, kEmitThreads, sizeof(EmitShared), &list_fits);
    prepare(k_emit<NSML_BF16, 2 * kEmitPer>, kEmitThreads, sizeof(EmitShared), &list_fits);
    prepare(k_select_small<NSML_F32, 1>, kSmallThreads, kSmallOneBlock * 4, &list_fits);
    prepare(k_select_small<NSML_BF16, 1>, kSmallThreads, kSmallOneBlock * 4, &list_fits);
    prepare(k_select_small<NSML_F32, kSmallBlocks>, kSmallThreads, kSmallPerBlock * 4, &list_fits);
    prepare(k_select_small<NSML_BF16, kSmallBlocks>, kSmallThreads, kSmallPerBlock * 4, &list_fits);
    prepare(k_sample<NSML_F32>, kSampleThreads, 0, &list_fits);
    prepare(k_sample<NSML_BF16>, kSampleThreads, 0, &list_fits);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&d.merge_small, k_merge<kDenseTileSmall>, kMergeThreads, 0);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&d.merge_large, k_merge<kDenseTileLarge>, kMergeThreads, 0);
    // The norm runs as one wave of resident blocks (a second, partial wave would read with a
    // fraction of the SMs' loads in flight).
    auto resident = [&](auto kernel, int* out) {
      int r = 0;
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, kernel, kCta, 0);
      if (*out == 0 || r < *out) *out = r;
    };
    resident(k_sumsq<NSML_F32>, &d.sumsq);
    resident(k_sumsq<NSML_BF16>, &d.sumsq);
    if (e == cudaSuccess && d.sumsq < 1) e = cudaErrorUnknown;
    int coop = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e != cudaSuccess || d.grid < 1 || list_fits < 1 || d.merge_small < 1 || d.merge_large < 1 || !coop) {
      return cuda_error();
    }
    d.ready = true;
  }
  *out = &d;
  return NSML_OK;
}

static inline bool valid_bits(int bits) { return bits == NSML_BITS_INT8 || bits == NSML_BITS_FP16 || bits == NSML_BITS_FP32; }
static inline bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

static inline unsigned int grid_for(unsigned long long work_items, unsigned long long per_block, int cap) {
  unsigned long long blocks = (work_items + per_block - 1) / per_block;
  if (blocks < 1) blocks = 1;
  if (blocks > (unsigned long long)cap) blocks = cap;
  return (unsigned int)blocks;
}

// The short, latency-bound kernels (sample, clear, list stage, small select, mask finish, partition) are launched at the
// highest stream priority.  When several buckets are in flight on several streams, every bucket pass that is ready sits in
// front of the device's block scheduler with thousands of blocks to place; a list-stage kernel that becomes
// ready later is otherwise placed only after all of them, so the passes of a step ran first, back to back,
// and the list stages afterwards with nothing to overlap them (measured with a timer in every kernel, before the list
// stage was rebuilt: 250 us of an 800 us step).  At high priority its few blocks are placed as soon as blocks of the running pass
// retire, and it runs beside the next pass.
static int high_priority() {
  static const int p = [] {
    int least = 0, greatest = 0;
    return cudaDeviceGetStreamPriorityRange(&least, &greatest) == cudaSuccess ? greatest : 0;
  }();
  return p;
}

template <class... KArgs, class... Args>
static cudaError_t launch_prio(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool cooperative,
                               unsigned int cluster_x, bool high, bool dependent, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[4];
  unsigned int na = 0;
  attr[na].id = cudaLaunchAttributePriority;
  attr[na].val.priority = high ? high_priority() : 0;
  ++na;
  if (cooperative) {
    attr[na].id = cudaLaunchAttributeCooperative;
    attr[na].val.cooperative = 1;
    ++na;
  }
  if (cluster_x) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = cluster_x;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
  }
  if (dependent) {  // may start while its predecessor in the stream still runs (programmatic dependent launch); the
                    // kernel calls pdl_wait before it touches anything the predecessor writes
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// without any attribute: at the priority of the stream
template <class... KArgs, class... Args>
static cudaError_t launch_plain(void (*kernel)(KArgs...), unsigned int grid, unsigned int block, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

static int64_t k_of(int64_t n, double ratio) {
  if (n < 1 || n > NSML_MAX_N || !(ratio > 0.0) || !(ratio <= 1.0)) return 0;
  double kd = std::ceil(ratio * (double)n);
  int64_t k = (int64_t)kd;
  if (k < 1) k = 1;
  if (k > n) k = n;
  return k;
}

// nsml_set_list_block_candidates: up to the default a block of the list stage per chunk of a short list, above it few.
constexpr int kListBlockCandidates = 4096;  // default of the knob
constexpr double kListFewBlocks = 10;       // blocks for a short list where the knob is well above it
static std::atomic<int> g_list_block_candidates{kListBlockCandidates};

// whether the caller has said that other calls fill the GPU
static bool many_calls() { return g_list_block_candidates.load(std::memory_order_relaxed) > kListBlockCandidates; }

static unsigned int grid_blocks(const DeviceInfo& dev) { return (unsigned int)(dev.sms < kGridMaxBlocks ? dev.sms / 2 * 2 : kGridMaxBlocks); }

// Small mode: the whole bucket is held in the shared memory of one block or cluster.
static bool use_small(int64_t n) { return n <= kSmallMaxN; }

// DTYPE: element type of `grad` (what the sample and the bucket pass read).  FDTYPE: element type of the
// bucket the later stages re-read; with a residual (local accumulation fused into the pass) that bucket is the residual buffer, float32, which then holds gradient + residual.
template <int DTYPE, int FDTYPE>
static int launch_compress(const void* grad, float* residual, const uint32_t* mask, int64_t n, int64_t k, int bits,
                           unsigned char* ws, unsigned char* payload, const CompressLayout& L, const PayloadLayout& P,
                           const DeviceInfo& dev, cudaStream_t st, bool keep_status = false) {
  Ctl* ctl = reinterpret_cast<Ctl*>(ws);
  BucketSrc<DTYPE> src{grad, mask};
  BucketSrc<FDTYPE> fsrc{residual != nullptr ? static_cast<const void*>(residual) : grad, mask};
  const unsigned long long tile = tile_elems<FDTYPE>();
  FinalizeParams fp;
  fp.n = (unsigned long long)n;
  fp.k = (unsigned long long)k;
  fp.bits = bits;
  fp.ctl = ctl;
  fp.hist = reinterpret_cast<unsigned int*>(ws + L.hist);
  fp.tiles = (unsigned int)(((unsigned long long)n + tile - 1) / tile);
  fp.list.off = reinterpret_cast<unsigned short*>(ws + L.cand_off);
  fp.list.val = reinterpret_cast<uint32_t*>(ws + L.cand_val);
  fp.list.tile_count = reinterpret_cast<unsigned int*>(ws + L.tile_count);
  fp.list.group_count = reinterpret_cast<unsigned int*>(ws + L.group_count);
  fp.list.window_hist = fp.hist + 3 * kMaxBins;
  fp.list.group_shift = group_shift_of(fp.tiles);
  fp.list.bins = reinterpret_cast<uint2*>(ws + L.bins);
  fp.list.bin_room = bin_room_of(n);
  const size_t chunks = align_up((size_t)n, tile_elems<NSML_BF16>()) / kChunk;
  fp.list.chunk_sum[0] = reinterpret_cast<unsigned long long*>(ws + L.chunk_sum);
  fp.list.chunk_sum[1] = fp.list.chunk_sum[0] + chunks;
  fp.list.block_fill = reinterpret_cast<unsigned int*>(ws + L.block_fill);
  fp.raw_val = reinterpret_cast<float*>(ws + L.raw_val);
  fp.residual = residual;
  fp.payload = payload;
  fp.P = P;
  cudaError_t le;
  if (use_small(n)) {
    LaunchScope scope(K_SELECT_SMALL, st);
    const bool one = n <= (int64_t)kSmallOneBlock;
    const unsigned int blocks = one ? 1 : kSmallBlocks;
    const unsigned int per_block = (unsigned int)align_up(((size_t)n + blocks - 1) / blocks, 128);
    auto kernel = one ? k_select_small<DTYPE, 1> : k_select_small<DTYPE, kSmallBlocks>;
    le = launch_prio(kernel, dim3(blocks), dim3(kSmallThreads), (size_t)per_block * 4, st, false, one ? 0 : kSmallBlocks, true, true, src, fp,
                     per_block, keep_status ? 1 : 0);
    return le == cudaSuccess ? NSML_OK : cuda_error();
  }
  // Dense mode: the select runs over the bucket itself, with no candidate list.
  if (const GridPlan g = grid_plan<FDTYPE>(n, k, DTYPE, grid_blocks(dev), many_calls(), residual != nullptr); g.grid != 0) {
    {
      LaunchScope scope(K_CLEAR, st);
      le = launch_prio(k_clear, dim3(8), dim3(kCta), 0, st, false, 0, true, true, reinterpret_cast<uint4*>(ws), (unsigned int)(L.zero_bytes / 16),
                       keep_status ? 1 : 0);
      if (le != cudaSuccess) return cuda_error();
    }
    LaunchScope scope(K_SELECT_GRID, st);
    // cooperative: every block co-resident; normal priority, it streams the whole bucket
    le = launch_prio(grid_kernel<DTYPE>(residual != nullptr, mask != nullptr, g.large), dim3(g.grid), dim3(kGridThreads), g.smem, st, true, 0, false,
                     true, src, fp, g.segs, g.rows, g.cap, g.room, g.rank_lo, g.rank_hi);
    return le == cudaSuccess ? NSML_OK : cuda_error();
  }
  const SamplePlan plan = sample_plan(n, k, DTYPE);
  {
    LaunchScope scope(K_SAMPLE, st);  // one cluster of kSampleBlocks blocks (the cluster shape is part of the kernel's definition)
    le = launch_prio(k_sample<DTYPE>, dim3(kSampleBlocks), dim3(kSampleThreads), 0, st, false, 0, true, true, src, residual,
                     (unsigned long long)n, plan.rank_lo, plan.rank_hi, ctl, reinterpret_cast<uint4*>(ws),
                     (unsigned int)(L.zero_bytes / 16), keep_status ? 1 : 0);
    if (le != cudaSuccess) return cuda_error();
  }
  {
    LaunchScope scope(K_COMPACT_BUCKET, st);  // a block per tile
    const bool fb = residual != nullptr, masked = mask != nullptr;
    le = launch_prio(fb ? (masked ? k_compact_bucket<DTYPE, true, true> : k_compact_bucket<DTYPE, true, false>)
                        : (masked ? k_compact_bucket<DTYPE, false, true> : k_compact_bucket<DTYPE, false, false>),
                     dim3(fp.tiles), dim3(kCta), 0, st, false, 0, false, true, src, residual, (unsigned long long)n, ctl, fp.list);
    if (le != cudaSuccess) return cuda_error();
  }
  {
    // Blocks draw chunks of the list by ticket, so the grid is free.  For a call that has the GPU to itself a block per
    // chunk, at most two per SM, is fastest (more would find no chunk).  A knob above the default says that other calls
    // fill the GPU: a block that waits for memory then holds what their passes need, so short lists get a few blocks
    // that take many chunks each and long ones one block per SM.  25M-element buckets, eight streams, knob 8192, ms per
    // step with 2 / 5 / 10 / 20 / 40 / 80 / 148 blocks: kept fraction 0.001 (2 buckets, 2 workers) 0.115 / 0.112 / 0.109
    // / 0.110 / 0.112 / 0.116 / 0.124, 0.003 0.133 / 0.122 / 0.121 / 0.118 / 0.119 / 0.124 / 0.131, 0.01 (5 buckets, 4
    // workers) 0.698 / 0.631 / 0.630 / 0.638 / 0.645 / 0.678 / 0.731: kListFewBlocks is near the best of all three.  A
    // block per 32768 candidates alone (the fourth power of the excess at 8192) is right at 0.01 only (two blocks at 0.001).
    // Long lists, 0.1: 1.14 / 0.549 / 0.382 / 0.363 / 0.357 / 0.352 / 0.355, with 296 0.378.
    LaunchScope scope(K_EMIT, st);
    const bool short_list = plan.expected <= 2.0 * dev.sms * kChunk;
    const double over = (double)g_list_block_candidates.load(std::memory_order_relaxed) / kListBlockCandidates;
    // a block per chunk, a quarter more where the GPU is the call's own: the list may be longer than expected, and a block
    // that has to take a second chunk makes the stage a third longer (25M elements with a residual at 0.01, timed in turn:
    // 100.7 -> 97.3 us)
    double want = plan.expected * (over > 1.0 ? 1.0 : 1.25) / kChunk + 1.0;
    if (over > 1.0 && short_list && want > kListFewBlocks) {
      want /= over * over * over * over;
      if (want < kListFewBlocks) want = kListFewBlocks;
    }
    const unsigned int cap = (over > 1.0 ? 1u : 2u) * dev.sms;
    const unsigned int grid = want < (double)cap ? (unsigned int)want : cap;
    // long lists: larger chunks, a block takes several
    le = launch_prio(short_list ? k_emit<FDTYPE, kEmitPer> : k_emit<FDTYPE, 2 * kEmitPer>, dim3(grid), dim3(kEmitThreads), sizeof(EmitShared), st, false, 0, true, true, fsrc, fp);
    if (le != cudaSuccess) return cuda_error();
  }
  return NSML_OK;
}

static int compress_impl(const void* grad, int64_t n, int grad_dtype, double ratio, int bits,
                         const uint32_t* prune_mask, void* payload, size_t payload_capacity, void* workspace,
                         size_t workspace_bytes, cudaStream_t st, bool keep_status = false) {
  if (grad == nullptr || payload == nullptr || workspace == nullptr) return NSML_ERR_ARG;
  if (grad_dtype != NSML_F32 && grad_dtype != NSML_BF16) return NSML_ERR_ARG;
  if (!valid_bits(bits)) return NSML_ERR_ARG;
  const int64_t k = k_of(n, ratio);
  if (k == 0) return NSML_ERR_ARG;
  if (!aligned(grad, 16) || !aligned(payload, 16) || !aligned(workspace, 256)) return NSML_ERR_ARG;
  if (prune_mask != nullptr && !aligned(prune_mask, 4)) return NSML_ERR_ARG;
  const PayloadLayout P = payload_layout(k, bits);
  const CompressLayout L = compress_layout(n);
  if (payload_capacity < P.total || workspace_bytes < L.total) return NSML_ERR_CAPACITY;
  const DeviceInfo* dev = nullptr;
  int rc = device_info(&dev);
  if (rc != NSML_OK) return rc;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  unsigned char* pl = static_cast<unsigned char*>(payload);
  if (grad_dtype == NSML_F32) rc = launch_compress<NSML_F32, NSML_F32>(grad, nullptr, prune_mask, n, k, bits, ws, pl, L, P, *dev, st, keep_status);
  else rc = launch_compress<NSML_BF16, NSML_BF16>(grad, nullptr, prune_mask, n, k, bits, ws, pl, L, P, *dev, st, keep_status);
  if (rc != NSML_OK) return rc;
  return NSML_OK;
}

// payload_bytes: sizes of the buffers behind the payload pointers, or nullptr when the caller does not
// know them.  timed: whether the launches may be bracketed by profiling events.
static int accumulate_impl(const void* const* payloads, const size_t* payload_bytes, int W, float* dense, int64_t n,
                           int zero_first, void* workspace, size_t workspace_bytes, cudaStream_t st, bool timed = true) {
  if (payloads == nullptr || dense == nullptr || workspace == nullptr) return NSML_ERR_ARG;
  if (W < 1 || W > NSML_MAX_WORKERS || n < 1 || n > NSML_MAX_N) return NSML_ERR_ARG;
  if (!aligned(dense, 16) || !aligned(workspace, 256)) return NSML_ERR_ARG;
  PayloadTable table;
  std::memset(&table, 0, sizeof(table));
  for (int w = 0; w < W; ++w) {
    if (payloads[w] == nullptr || !aligned(payloads[w], 16)) return NSML_ERR_ARG;
    table.p[w] = static_cast<const unsigned char*>(payloads[w]);
    if (payload_bytes != nullptr) {
      if (payload_bytes[w] < sizeof(nsml_payload_header)) return NSML_ERR_ARG;
      table.bytes[w] = payload_bytes[w];
    }
  }
  const AccumulateLayout L = accumulate_layout(n, W);
  if (workspace_bytes < L.total) return NSML_ERR_CAPACITY;
  const DeviceInfo* dev = nullptr;
  int rc = device_info(&dev);
  if (rc != NSML_OK) return rc;

  unsigned char* ws = static_cast<unsigned char*>(workspace);
  int* status = reinterpret_cast<int*>(ws);
  unsigned int* offsets = reinterpret_cast<unsigned int*>(ws + L.offsets);
  const unsigned int tile = (unsigned int)dense_tile(n);
  const unsigned int tiles = (unsigned int)((n + tile - 1) / tile);
  unsigned long long largest = 0;  // payload, in bytes; 0 = not known
  for (int w = 0; w < W; ++w) largest = table.bytes[w] > largest ? table.bytes[w] : largest;
  cudaError_t le;
  {
    LaunchScope scope(K_PARTITION, st, timed);  // also clears the status word
    // (where many calls are in flight, blocks that wait for the kernel before them would hold what the others need)
    const bool many = many_calls();
    le = launch_prio(k_partition, dim3(partition_blocks(n, tiles, W, largest, many), W), dim3(kPartBounds), 0, st, false, 0, true, !many, table, W, (unsigned long long)n,
                tiles, tile == kDenseTileLarge ? 13u : 11u, offsets, status);
    if (le != cudaSuccess) return cuda_error();
  }
  {
    LaunchScope scope(K_MERGE, st, timed);
    const bool large = tile == kDenseTileLarge;
    const unsigned int grid = grid_for(tiles, 1, dev->sms * (large ? dev->merge_large : dev->merge_small));
    auto kernel = large ? k_merge<kDenseTileLarge> : k_merge<kDenseTileSmall>;
    le = launch_prio(kernel, dim3(grid), dim3(kMergeThreads), 0, st, false, 0, false, true, table, W, dense, (unsigned long long)n, zero_first, tiles, offsets, status);
    if (le != cudaSuccess) return cuda_error();
  }
  return NSML_OK;
}

// ---- Alg. 2 Step 1: L2 norm and gate ----------------------------------------
// Blocks of the streaming kernels of nsml_adaptive.cuh: enough to keep every SM's loads in flight.
static unsigned int stream_grid(int64_t n, const DeviceInfo& dev, int per_sm, unsigned int cap) {
  unsigned int g = grid_for(((unsigned long long)n + kStreamTile - 1) / kStreamTile, 1, dev.sms * per_sm);
  return g < cap ? g : cap;
}

static int sumsq_impl(const void* grad, int64_t n, int grad_dtype, void* workspace, size_t workspace_bytes,
                      cudaStream_t st, SumsqCtl* to_host = nullptr) {
  if (grad == nullptr || workspace == nullptr) return NSML_ERR_ARG;
  if (grad_dtype != NSML_F32 && grad_dtype != NSML_BF16) return NSML_ERR_ARG;
  if (n < 1 || n > NSML_MAX_N) return NSML_ERR_ARG;
  if (!aligned(grad, 16) || !aligned(workspace, 256)) return NSML_ERR_ARG;
  if (workspace_bytes < kSumsqWorkspace) return NSML_ERR_CAPACITY;
  const DeviceInfo* dev = nullptr;
  int rc = device_info(&dev);
  if (rc != NSML_OK) return rc;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  if (cudaMemsetAsync(ws, 0, 256, st) != cudaSuccess) return cuda_error();
  SumsqCtl* ctl = reinterpret_cast<SumsqCtl*>(ws);
  double* partials = reinterpret_cast<double*>(ws + 256);
  const unsigned int grid = stream_grid(n, *dev, dev->sumsq < 8 ? dev->sumsq : 8, kSumsqMaxBlocks);
  {
    LaunchScope scope(K_SUMSQ, st);
    cudaError_t le;
    if (grad_dtype == NSML_F32)
      le = launch_plain(k_sumsq<NSML_F32>, grid, kCta, st, BucketSrc<NSML_F32>{grad, nullptr}, (unsigned long long)n, ctl, partials, to_host);
    else
      le = launch_plain(k_sumsq<NSML_BF16>, grid, kCta, st, BucketSrc<NSML_BF16>{grad, nullptr}, (unsigned long long)n, ctl, partials, to_host);
    if (le != cudaSuccess) return cuda_error();
  }
  return NSML_OK;
}

// A few bytes of page-locked host memory that kernels of any device can write; one per calling thread, freed with it.
struct HostSlot {
  SumsqCtl* at = nullptr;
  HostSlot() {
    // (allowed while another thread captures a stream)
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    if (cudaThreadExchangeStreamCaptureMode(&mode) != cudaSuccess) return;
    void* p = nullptr;
    if (cudaHostAlloc(&p, sizeof(SumsqCtl), cudaHostAllocPortable | cudaHostAllocMapped) == cudaSuccess) at = static_cast<SumsqCtl*>(p);
    else cudaGetLastError();
    cudaThreadExchangeStreamCaptureMode(&mode);
  }
  ~HostSlot() { if (at != nullptr) cudaFreeHost(at); }
};

// Sum of squares, waited for: synchronises the stream.
static int sumsq_wait(const void* grad, int64_t n, int grad_dtype, void* workspace, size_t workspace_bytes, cudaStream_t st,
                      double* sumsq) {
  static thread_local HostSlot slot;
  const int rc = sumsq_impl(grad, n, grad_dtype, workspace, workspace_bytes, st, slot.at);
  if (rc != NSML_OK) return rc;
  SumsqCtl pageable;
  SumsqCtl* host = slot.at;
  if (host == nullptr) {
    host = &pageable;
    if (cudaMemcpyAsync(host, workspace, sizeof(*host), cudaMemcpyDeviceToHost, st) != cudaSuccess) return cuda_error();
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) return cuda_error();
  if (host->status != NSML_OK) return host->status;
  *sumsq = host->sumsq;
  return NSML_OK;
}

static int gate(double ratio, double l2, double tr_q, double tr_d, int plain_bits, double* ratio_out, int* bits_out) {
  if (!(ratio > 0.0) || !(ratio <= 1.0) || !valid_bits(plain_bits) || !(l2 >= 0.0) || tr_q != tr_q || tr_d != tr_d)
    return NSML_ERR_ARG;
  if (ratio < tr_q && l2 > tr_d) {
    const double doubled = 2.0 * ratio;
    *ratio_out = doubled < 1.0 ? doubled : 1.0;
    *bits_out = NSML_BITS_FP16;
  } else {
    *ratio_out = ratio;
    *bits_out = plain_bits;
  }
  return NSML_OK;
}

// ---- Alg. 2 Step 2: pruning mask from the weights ---------------------------
static int64_t pruned_count(int64_t n, double ratio) {
  if (n < 1 || n > NSML_MAX_N || !(ratio > 0.0) || !(ratio <= 1.0)) return -1;
  const double rate = 0.5 * (1.0 - ratio);
  int64_t m = (int64_t)std::ceil(rate * (double)n);
  if (m < 0) m = 0;
  if (m > n) m = n;
  return m;
}

static int prune_impl(const float* weights, int64_t n, double ratio, uint32_t* mask, void* workspace,
                      size_t workspace_bytes, cudaStream_t st) {
  if (weights == nullptr || mask == nullptr || workspace == nullptr) return NSML_ERR_ARG;
  const int64_t m = pruned_count(n, ratio);
  if (m < 0) return NSML_ERR_ARG;
  if (!aligned(weights, 16) || !aligned(mask, 4) || !aligned(workspace, 256)) return NSML_ERR_ARG;
  const PruneLayout L = prune_layout(n);
  if (workspace_bytes < L.total) return NSML_ERR_CAPACITY;
  const DeviceInfo* dev = nullptr;
  int rc = device_info(&dev);
  if (rc != NSML_OK) return rc;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  if (m == 0) {  // ratio 1: nothing is pruned
    if (cudaMemsetAsync(ws, 0, 256, st) != cudaSuccess) return cuda_error();
    if (cudaMemsetAsync(mask, 0, (size_t)((n + 31) / 32) * 4, st) != cudaSuccess) return cuda_error();
    return NSML_OK;
  }
  Ctl* ctl = reinterpret_cast<Ctl*>(ws);
  uint2* list = reinterpret_cast<uint2*>(ws + L.list);
  const BucketSrc<NSML_F32> src{weights, nullptr};
  const bool sampled = n >= (int64_t)kSamples;
  cudaError_t le;
  if (sampled) {
    // bracket of the (n - m + 1)-th largest magnitude; also clears the control block and the histograms
    const SamplePlan plan = sample_plan(n, n - m + 1, NSML_F32);
    {
      LaunchScope scope(K_SAMPLE, st);
      le = launch_prio(k_sample<NSML_F32>, dim3(kSampleBlocks), dim3(kSampleThreads), 0, st, false, 0, true, true, src, nullptr,
                       (unsigned long long)n, plan.rank_lo, plan.rank_hi, ctl, reinterpret_cast<uint4*>(ws), (unsigned int)(L.zero_bytes / 16), 0);
      if (le != cudaSuccess) return cuda_error();
    }
    LaunchScope scope(K_PRUNE_PASS, st);
    le = launch_prio(k_prune_pass, dim3((unsigned int)((n + kPruneTile - 1) / kPruneTile)), dim3(kCta), 0, st, false, 0, false, true, src,
                     (unsigned long long)n, ctl, list, (unsigned int)L.cap, mask);
    if (le != cudaSuccess) return cuda_error();
  } else if (cudaMemsetAsync(ws, 0, L.zero_bytes, st) != cudaSuccess) {
    return cuda_error();
  }
  {
    LaunchScope scope(K_PRUNE_FINISH, st);
    const unsigned int grid = grid_for((unsigned long long)n, kPruneUnit, 2 * dev->sms);
    le = launch_prio(k_prune_finish, dim3(grid), dim3(kPruneThreads), 0, st, false, 0, true, sampled, src, (unsigned int)n, (unsigned int)m, ctl,
                     reinterpret_cast<unsigned int*>(ws + L.hist), list, (unsigned int)L.cap, reinterpret_cast<uint2*>(ws + L.bin_list),
                     reinterpret_cast<unsigned int*>(ws + L.unit_ties), mask, sampled ? 1 : 0);
    if (le != cudaSuccess) return cuda_error();
  }
  return NSML_OK;
}

// ---- Section 4.2 Step 3: local accumulation of the filtered gradients ---------
static int feedback_impl(const void* grad, float* residual, int64_t n, int grad_dtype, double ratio, int bits,
                         const uint32_t* prune_mask, void* payload, size_t payload_capacity, void* workspace,
                         size_t workspace_bytes, cudaStream_t st) {
  if (grad == nullptr || residual == nullptr) return NSML_ERR_ARG;
  if (grad_dtype != NSML_F32 && grad_dtype != NSML_BF16) return NSML_ERR_ARG;
  const int64_t k = k_of(n, ratio);
  if (k == 0 || !valid_bits(bits)) return NSML_ERR_ARG;
  if (!aligned(grad, 16) || !aligned(residual, 16)) return NSML_ERR_ARG;
  if (payload == nullptr || workspace == nullptr || !aligned(payload, 16) || !aligned(workspace, 256)) return NSML_ERR_ARG;
  if (payload_capacity < payload_layout(k, bits).total || workspace_bytes < compress_layout(n).total)
    return NSML_ERR_CAPACITY;
  const DeviceInfo* dev = nullptr;
  int rc = device_info(&dev);
  if (rc != NSML_OK) return rc;
  // the kernels that read the gradient add the residual to it, leave the sum there and take out what the payload carries
  if (prune_mask != nullptr && !aligned(prune_mask, 4)) return NSML_ERR_ARG;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  unsigned char* pl = static_cast<unsigned char*>(payload);
  const PayloadLayout P = payload_layout(k, bits);
  const CompressLayout L = compress_layout(n);
  if (grad_dtype == NSML_F32)
    rc = launch_compress<NSML_F32, NSML_F32>(grad, residual, prune_mask, n, k, bits, ws, pl, L, P, *dev, st);
  else
    rc = launch_compress<NSML_BF16, NSML_F32>(grad, residual, prune_mask, n, k, bits, ws, pl, L, P, *dev, st);
  if (rc != NSML_OK) return rc;
  return NSML_OK;
}

// ---- scratch for nsml_decompress_accumulate_static --------------------------
// Part of the library image: every device that loads the library holds this
// array until exit.  In host code the name below is only a handle; the device
// address is looked up once per device with cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_static_scratch[NSML_STATIC_SCRATCH_BYTES];

static void* g_static_scratch_addr[64];
static std::mutex g_static_mutex;

static int static_scratch(void** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cuda_error();
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (g_static_scratch_addr[dev] == nullptr) {
    void* addr = nullptr;
    if (cudaGetSymbolAddress(&addr, g_static_scratch) != cudaSuccess || addr == nullptr) {
      return cuda_error();
    }
    g_static_scratch_addr[dev] = addr;
  }
  *out = g_static_scratch_addr[dev];
  return NSML_OK;
}

}  // namespace nsml

using namespace nsml;

extern "C" {

int64_t nsml_k_of(int64_t n, double ratio) { return k_of(n, ratio); }

int nsml_compress_strategy(int64_t n, double ratio) { return nsml_compress_strategy_of(n, ratio, NSML_F32, 0); }

int nsml_compress_strategy_of(int64_t n, double ratio, int grad_dtype, int residual) {
  const int64_t k = k_of(n, ratio);
  if (k == 0 || (grad_dtype != NSML_F32 && grad_dtype != NSML_BF16)) return NSML_ERR_ARG;
  const DeviceInfo* dev = nullptr;
  const int rc = device_info(&dev);
  if (rc != NSML_OK) return rc;
  const unsigned int blocks = grid_blocks(*dev);
  const GridPlan g = grad_dtype == NSML_F32 || residual ? grid_plan<NSML_F32>(n, k, grad_dtype, blocks, many_calls(), residual != 0)
                                                        : grid_plan<NSML_BF16>(n, k, grad_dtype, blocks, many_calls());
  return g.grid != 0 ? NSML_STRATEGY_DENSE : NSML_STRATEGY_LIST;
}

int nsml_set_list_block_candidates(int candidates) {
  if (candidates < 1024 || candidates > 8192) return NSML_ERR_ARG;
  g_list_block_candidates.store(candidates, std::memory_order_relaxed);
  return NSML_OK;
}

size_t nsml_payload_bytes(int64_t n, double ratio, int bits) {
  if (!valid_bits(bits)) return 0;
  const int64_t k = k_of(n, ratio);
  if (k == 0) return 0;
  return payload_layout(k, bits).total;
}

size_t nsml_workspace_bytes(int64_t n, int grad_dtype) {
  if (n < 1 || n > NSML_MAX_N || (grad_dtype != NSML_F32 && grad_dtype != NSML_BF16)) return 0;
  return compress_layout(n).total;
}

size_t nsml_accumulate_workspace_bytes(int64_t n, int W) {
  if (n < 1 || n > NSML_MAX_N || W < 1 || W > NSML_MAX_WORKERS) return 0;
  return accumulate_layout(n, W).ask;
}

int nsml_compress(const void* grad, int64_t n, int grad_dtype, double ratio, int bits, const uint32_t* prune_mask,
                  void* payload, size_t payload_capacity, void* workspace, size_t workspace_bytes, void* stream) {
  return compress_impl(grad, n, grad_dtype, ratio, bits, prune_mask, payload, payload_capacity, workspace,
                       workspace_bytes, static_cast<cudaStream_t>(stream));
}

int nsml_decompress_accumulate(const void* const* payloads, int W, float* dense, int64_t n, int zero_first,
                               void* workspace, size_t workspace_bytes, void* stream) {
  return accumulate_impl(payloads, nullptr, W, dense, n, zero_first, workspace, workspace_bytes,
                         static_cast<cudaStream_t>(stream));
}

int nsml_decompress_accumulate_sized(const void* const* payloads, const size_t* payload_bytes, int W, float* dense,
                                     int64_t n, int zero_first, void* workspace, size_t workspace_bytes, void* stream) {
  if (payload_bytes == nullptr) return NSML_ERR_ARG;
  return accumulate_impl(payloads, payload_bytes, W, dense, n, zero_first, workspace, workspace_bytes,
                         static_cast<cudaStream_t>(stream));
}

int nsml_decompress_accumulate_static(const void* const* payloads, int W, float* dense, int64_t n, int zero_first,
                                      void* stream, int* status_out) {
  if (n > NSML_STATIC_MAX_N || W > NSML_STATIC_MAX_WORKERS) return NSML_ERR_CAPACITY;
  if (n < 1 || W < 1) return NSML_ERR_ARG;
  if (accumulate_layout(n, W).total > (size_t)NSML_STATIC_SCRATCH_BYTES) return NSML_ERR_CAPACITY;
  void* scratch = nullptr;
  int rc = static_scratch(&scratch);
  if (rc != NSML_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  rc = accumulate_impl(payloads, nullptr, W, dense, n, zero_first, scratch, NSML_STATIC_SCRATCH_BYTES, st, /*timed=*/false);
  if (rc != NSML_OK || status_out == nullptr) return rc;
  int value = 0;
  if (cudaMemcpyAsync(&value, scratch, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return cuda_error();
  if (cudaStreamSynchronize(st) != cudaSuccess) return cuda_error();
  *status_out = value;
  return NSML_OK;
}

// ---- Alg. 2 Steps 1-2 and the local accumulation of Step 3 --------------------
size_t nsml_l2_workspace_bytes(void) { return kSumsqWorkspace; }

int nsml_grad_l2(const void* grad, int64_t n, int grad_dtype, void* workspace, size_t workspace_bytes, void* stream,
                 double* l2_out) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (l2_out == nullptr) return sumsq_impl(grad, n, grad_dtype, workspace, workspace_bytes, st);
  double sumsq = 0.0;
  const int rc = sumsq_wait(grad, n, grad_dtype, workspace, workspace_bytes, st, &sumsq);
  if (rc != NSML_OK) return rc;
  *l2_out = std::sqrt(sumsq);
  return NSML_OK;
}

int nsml_quantize_gate(double ratio, double l2, double tr_q, double tr_d, int plain_bits, double* ratio_out,
                       int* bits_out) {
  if (ratio_out == nullptr || bits_out == nullptr) return NSML_ERR_ARG;
  return gate(ratio, l2, tr_q, tr_d, plain_bits, ratio_out, bits_out);
}

int64_t nsml_pruned_count(int64_t n, double ratio) {
  const int64_t m = pruned_count(n, ratio);
  return m < 0 ? 0 : m;
}

size_t nsml_prune_workspace_bytes(int64_t n) {
  if (n < 1 || n > NSML_MAX_N) return 0;
  return prune_layout(n).total;
}

int nsml_prune_mask_build(const float* weights, int64_t n, double ratio, uint32_t* prune_mask, void* workspace,
                          size_t workspace_bytes, void* stream) {
  return prune_impl(weights, n, ratio, prune_mask, workspace, workspace_bytes, static_cast<cudaStream_t>(stream));
}

int nsml_compress_feedback(const void* grad, float* residual, int64_t n, int grad_dtype, double ratio, int bits,
                           const uint32_t* prune_mask, void* payload, size_t payload_capacity, void* workspace,
                           size_t workspace_bytes, void* stream) {
  return feedback_impl(grad, residual, n, grad_dtype, ratio, bits, prune_mask, payload, payload_capacity, workspace,
                       workspace_bytes, static_cast<cudaStream_t>(stream));
}

size_t nsml_adaptive_payload_bytes(int64_t n, double ratio, double tr_q, int plain_bits) {
  size_t need = nsml_payload_bytes(n, ratio, plain_bits);
  if (need == 0) return 0;
  if (ratio < tr_q) {
    const double doubled = 2.0 * ratio;
    const size_t q = nsml_payload_bytes(n, doubled < 1.0 ? doubled : 1.0, NSML_BITS_FP16);
    if (q > need) need = q;
  }
  return need;
}

size_t nsml_adaptive_workspace_bytes(int64_t n, int grad_dtype) {
  size_t need = nsml_workspace_bytes(n, grad_dtype);
  if (need == 0) return 0;
  if (need < kSumsqWorkspace) need = kSumsqWorkspace;
  const size_t p = prune_layout(n).total;
  return need < p ? p : need;
}

int nsml_compress_adaptive(const void* grad, int64_t n, int grad_dtype, double ratio, double tr_q, double tr_d,
                           int plain_bits, const float* weights, uint32_t* prune_mask, void* payload,
                           size_t payload_capacity, void* workspace, size_t workspace_bytes, void* stream,
                           double* ratio_used, int* bits_used, double* l2_out) {
  if (ratio_used == nullptr || bits_used == nullptr) return NSML_ERR_ARG;
  if (!(ratio > 0.0) || !(ratio <= 1.0) || !valid_bits(plain_bits) || tr_q != tr_q || tr_d != tr_d) return NSML_ERR_ARG;
  if (weights != nullptr && prune_mask == nullptr) return NSML_ERR_ARG;
  const size_t need_ws = nsml_adaptive_workspace_bytes(n, grad_dtype);
  if (need_ws == 0) return NSML_ERR_ARG;
  if (workspace_bytes < need_ws) return NSML_ERR_CAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // Step 1: the norm is needed only when the ratio is below the quantisation check threshold
  double use_ratio = ratio, l2 = -1.0;
  int use_bits = plain_bits;
  if (ratio < tr_q) {
    double sumsq = 0.0;
    int rc = sumsq_wait(grad, n, grad_dtype, workspace, workspace_bytes, st, &sumsq);
    if (rc != NSML_OK) return rc;
    l2 = std::sqrt(sumsq);
    rc = gate(ratio, l2, tr_q, tr_d, plain_bits, &use_ratio, &use_bits);
    if (rc != NSML_OK) return rc;
  }
  if (l2_out != nullptr) *l2_out = l2;
  *ratio_used = use_ratio;
  *bits_used = use_bits;
  // Step 2: the mask follows the ratio Step 1 left
  if (weights != nullptr) {
    const int rc = prune_impl(weights, n, use_ratio, prune_mask, workspace, workspace_bytes, st);
    if (rc != NSML_OK) return rc;
  }
  // Step 3.  The mask build shares the workspace and its status word with this step: when it ran, the
  // word is kept instead of cleared, so that non-finite weights found in Step 2 are still reported.
  return compress_impl(grad, n, grad_dtype, use_ratio, use_bits, prune_mask, payload, payload_capacity, workspace,
                       workspace_bytes, st, /*keep_status=*/weights != nullptr);
}

// ---- host-buffer variants --------------------------------------------------
static size_t elem_size(int grad_dtype) { return grad_dtype == NSML_F32 ? 4 : 2; }

size_t nsml_compress_host_scratch_bytes(int64_t n, int grad_dtype, double ratio, int bits) {
  const size_t ws = nsml_workspace_bytes(n, grad_dtype);
  const size_t pb = nsml_payload_bytes(n, ratio, bits);
  if (ws == 0 || pb == 0) return 0;
  return align_up(ws, 256) + align_up((size_t)n * elem_size(grad_dtype), 256) +
         align_up((size_t)((n + 31) / 32) * 4, 256) + align_up(pb, 256);
}

int nsml_compress_host(const void* grad_host, int64_t n, int grad_dtype, double ratio, int bits,
                       const uint32_t* prune_mask_host, void* payload_host, size_t payload_capacity,
                       void* device_scratch, size_t scratch_bytes, void* stream) {
  if (grad_host == nullptr || payload_host == nullptr || device_scratch == nullptr) return NSML_ERR_ARG;
  const size_t need = nsml_compress_host_scratch_bytes(n, grad_dtype, ratio, bits);
  if (need == 0 || !aligned(device_scratch, 256)) return NSML_ERR_ARG;
  const size_t pb = nsml_payload_bytes(n, ratio, bits);
  if (scratch_bytes < need || payload_capacity < pb) return NSML_ERR_CAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  unsigned char* base = static_cast<unsigned char*>(device_scratch);
  const size_t ws = align_up(nsml_workspace_bytes(n, grad_dtype), 256);
  const size_t gbytes = (size_t)n * elem_size(grad_dtype);
  const size_t mbytes = (size_t)((n + 31) / 32) * 4;
  unsigned char* d_grad = base + ws;
  unsigned char* d_mask = d_grad + align_up(gbytes, 256);
  unsigned char* d_payload = d_mask + align_up(mbytes, 256);
  if (cudaMemcpyAsync(d_grad, grad_host, gbytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return cuda_error();
  if (prune_mask_host != nullptr &&
      cudaMemcpyAsync(d_mask, prune_mask_host, mbytes, cudaMemcpyHostToDevice, st) != cudaSuccess)
    return cuda_error();
  int rc = compress_impl(d_grad, n, grad_dtype, ratio, bits,
                         prune_mask_host ? reinterpret_cast<const uint32_t*>(d_mask) : nullptr, d_payload, pb, base, ws,
                         st);
  if (rc != NSML_OK) return rc;
  if (cudaMemcpyAsync(payload_host, d_payload, pb, cudaMemcpyDeviceToHost, st) != cudaSuccess) return cuda_error();
  return NSML_OK;
}

size_t nsml_accumulate_host_scratch_bytes(int64_t n, int W, size_t total_payload_bytes) {
  const size_t ws = nsml_accumulate_workspace_bytes(n, W);
  if (ws == 0) return 0;
  return align_up(ws, 256) + align_up((size_t)n * 4, 256) + total_payload_bytes + (size_t)W * 256;
}

int nsml_decompress_accumulate_host(const void* const* payloads_host, const size_t* payload_bytes, int W,
                                    float* dense_host, int64_t n, int zero_first, void* device_scratch,
                                    size_t scratch_bytes, void* stream) {
  if (payloads_host == nullptr || payload_bytes == nullptr || dense_host == nullptr || device_scratch == nullptr)
    return NSML_ERR_ARG;
  if (W < 1 || W > NSML_MAX_WORKERS || !aligned(device_scratch, 256)) return NSML_ERR_ARG;
  if (n < 1 || n > NSML_MAX_N) return NSML_ERR_ARG;
  size_t total = 0;
  for (int w = 0; w < W; ++w) {
    if (payloads_host[w] == nullptr || payload_bytes[w] < sizeof(nsml_payload_header)) return NSML_ERR_ARG;
    // (the headers are not looked at here: a payload may still be on its way into host memory, written by an
    // earlier asynchronous call on this stream; the device checks every header against payload_bytes[w])
    total += payload_bytes[w];
  }
  const size_t need = nsml_accumulate_host_scratch_bytes(n, W, total);
  if (need == 0) return NSML_ERR_ARG;
  if (scratch_bytes < need) return NSML_ERR_CAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  unsigned char* base = static_cast<unsigned char*>(device_scratch);
  const size_t ws = align_up(nsml_accumulate_workspace_bytes(n, W), 256);
  float* d_dense = reinterpret_cast<float*>(base + ws);
  unsigned char* cursor = base + ws + align_up((size_t)n * 4, 256);
  const void* d_payloads[NSML_MAX_WORKERS];
  for (int w = 0; w < W; ++w) {
    if (cudaMemcpyAsync(cursor, payloads_host[w], payload_bytes[w], cudaMemcpyHostToDevice, st) != cudaSuccess)
      return cuda_error();
    d_payloads[w] = cursor;
    cursor += align_up(payload_bytes[w], 256);
  }
  if (!zero_first &&
      cudaMemcpyAsync(d_dense, dense_host, (size_t)n * 4, cudaMemcpyHostToDevice, st) != cudaSuccess)
    return cuda_error();
  int rc = accumulate_impl(d_payloads, payload_bytes, W, d_dense, n, zero_first, base, ws, st);
  if (rc != NSML_OK) return rc;
  if (cudaMemcpyAsync(dense_host, d_dense, (size_t)n * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return cuda_error();
  return NSML_OK;
}

int nsml_last_status(const void* workspace, void* stream, int* status_out) {
  if (workspace == nullptr || status_out == nullptr) return NSML_ERR_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int value = 0;
  if (cudaMemcpyAsync(&value, workspace, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return cuda_error();
  if (cudaStreamSynchronize(st) != cudaSuccess) return cuda_error();
  *status_out = value;
  return NSML_OK;
}

int nsml_selftest_bounded_wait(void* workspace, size_t workspace_bytes, int max_polls, void* stream) {
  if (workspace == nullptr || !aligned(workspace, 256) || max_polls < 1 || max_polls > (1 << 16)) return NSML_ERR_ARG;
  if (workspace_bytes < 256) return NSML_ERR_CAPACITY;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(workspace, 0, 256, st) != cudaSuccess) return cuda_error();
  if (launch_plain(k_barrier_probe, 2, 32, st, static_cast<Ctl*>(workspace), max_polls) != cudaSuccess) return cuda_error();
  return NSML_OK;
}

const char* nsml_strerror(int status) {
  switch (status) {
    case NSML_OK: return "ok";
    case NSML_ERR_ARG: return "bad argument (null or misaligned pointer, size or enum out of range)";
    case NSML_ERR_CAPACITY: return "payload buffer or workspace too small";
    case NSML_ERR_CUDA: return "a CUDA runtime call failed";
    case NSML_ERR_NONFINITE: return "the gradient bucket holds NaN or Inf";
    case NSML_ERR_TIMEOUT: return "a bounded wait between thread blocks ran out";
    case NSML_ERR_PAYLOAD: return "payload header or index out of range";
    case NSML_ERR_INTERNAL: return "internal invariant failed: survivor count differs from k";
    default: return "unknown status";
  }
}

// ---- instrumentation -------------------------------------------------------
int nsml_kernel_count(void) { return K_COUNT; }

const char* nsml_kernel_name(int kernel_id) {
  return (kernel_id >= 0 && kernel_id < K_COUNT) ? kKernelNames[kernel_id] : "";
}

int64_t nsml_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

int nsml_prof_enable(int on) {
  std::lock_guard<std::mutex> lock(g_prof_mutex);
  if (!on) {
    for (ProfRecord& r : g_prof_records) {
      cudaEventDestroy(r.start);
      cudaEventDestroy(r.stop);
    }
    g_prof_records.clear();
  }
  g_prof_on.store(on != 0, std::memory_order_relaxed);
  return NSML_OK;
}

int nsml_prof_read(int kernel_id, double* total_ms, int64_t* launches) {
  if (kernel_id < 0 || kernel_id >= K_COUNT || total_ms == nullptr || launches == nullptr) return NSML_ERR_ARG;
  std::lock_guard<std::mutex> lock(g_prof_mutex);
  prof_drain_locked();
  *total_ms = g_prof_ms[kernel_id];
  *launches = g_prof_launches[kernel_id];
  return NSML_OK;
}

int nsml_prof_reset(void) {
  std::lock_guard<std::mutex> lock(g_prof_mutex);
  prof_drain_locked();
  for (int i = 0; i < K_COUNT; ++i) {
    g_prof_ms[i] = 0.0;
    g_prof_launches[i] = 0;
  }
  return NSML_OK;
}

}  // extern "C"
