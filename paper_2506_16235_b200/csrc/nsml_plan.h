// What a call is launched with, worked out on the host: the ranks the sample is asked for, and whether and how the grid
// select (nsml_grid.cuh) takes the call.  Plain C++, so that every size can be gone through without a GPU.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>

#include "nsml.h"

#ifdef __CUDACC__
#define NSML_HD __host__ __device__
#else
#define NSML_HD
#endif

namespace nsml {

NSML_HD inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ---- the sample ----
constexpr int kSamples = 16384;  // strata
template <int DTYPE>
NSML_HD constexpr int sample_keys() { return DTYPE == NSML_F32 ? 4 : 8; }  // keys per stratum: 16 bytes
inline double sampled_keys(int grad_dtype) { return (double)kSamples * (grad_dtype == NSML_F32 ? sample_keys<NSML_F32>() : sample_keys<NSML_BF16>()); }

// What the sample of a call is asked for: the ranks (from the top, 1-based) of the two sample keys `sigmas` standard
// deviations either side of the expected rank of the k-th largest, and the number of candidates to expect above
// the lower one.  rank_lo = 0: do not sample (small bucket, or nearly everything is kept).
struct SamplePlan {
  unsigned int rank_lo = 0, rank_hi = 0;
  double expected = 0.0;
};

inline SamplePlan sample_plan(int64_t n, int64_t k, int grad_dtype, double sigmas = 6.0) {
  SamplePlan s;
  if (n < (int64_t)kSamples) return s;
  const double keys = sampled_keys(grad_dtype);
  const double p = (double)k / (double)n, mean = keys * p, spread = sigmas * std::sqrt(keys * p * (1.0 - p));
  const double lo = std::ceil(mean + spread) + 1.0, hi = std::floor(mean - spread);
  if (lo < keys) s.rank_lo = (unsigned int)lo;
  // (the largest sampled key, with about n / keys elements above it, where that is safely fewer than k)
  s.rank_hi = hi >= 1.0 ? (unsigned int)hi : 8.0 * (double)n / keys < (double)k ? 1u : 0u;
  s.expected = (double)n * (mean + spread) / keys * 1.04 + 64.0;  // (the bound is rounded down to 14 key bits: a few per cent more)
  return s;
}

// ---- the grid select ----
constexpr int kGridThreads = 1024, kGridWarps = kGridThreads / 32;
constexpr int kGridMaxBlocks = 192;
constexpr size_t kGridSmem = 232448;          // 227 KB
constexpr size_t kGridSharedBytes = 24752;    // of GridShared
constexpr unsigned int kGridMaxCap = 384;     // window entries of a warp in shared memory, at most
constexpr double kGridListMargin = 1.25;      // ... and how many times as many as expected there has to be room for
constexpr int kGridPitch = kGridWarps + 1;    // words between the rows of the tables
constexpr unsigned int kGridSliceBytes = 512;

template <int VT>
NSML_HD constexpr unsigned int grid_seg() { return kGridThreads * (VT == NSML_F32 ? 4 : 8); }  // elements of a segment
// An entry's place in its warp's part of the bucket has 16 bits: the row and the offset inside the row's slice.
template <int VT>
NSML_HD constexpr int grid_off_bits() { return VT == NSML_F32 ? 7 : 8; }
template <int VT>
NSML_HD constexpr unsigned int grid_max_rows() { return 1u << (16 - grid_off_bits<VT>()); }
template <int VT>
NSML_HD constexpr unsigned int grid_slots() { return grid_seg<VT>() / NSML_QBLOCK + 1; }  // payload blocks of 1024 a segment can touch
template <int VT>
NSML_HD constexpr size_t grid_entry_bytes() { return VT == NSML_F32 ? 6 : 4; }  // of the window's list
// what of the shared memory a row takes: three tables, six words, the maxima (scales) of its payload blocks and their
// inverses, where its slices are
template <int VT>
NSML_HD constexpr size_t grid_row_bytes() { return (3 * kGridPitch + 6 + 2 * grid_slots<VT>()) * 4 + kGridWarps * 2; }
// cap: window entries a warp has room for; room: slices the block has room for.  (Tables and lists in the workspace: none
// of either here.)
template <int VT>
NSML_HD inline size_t grid_smem(unsigned int rows, unsigned int cap, unsigned int room) {
  return align_up(kGridSharedBytes + (size_t)rows * grid_row_bytes<VT>() + (size_t)kGridWarps * cap * grid_entry_bytes<VT>(), 16) +
         (size_t)room * kGridSliceBytes;
}

// Kept fraction from which the select runs over the bucket itself (k_select_grid) and not over a candidate list.  us, list /
// grid select, buckets of tensors of different scales | of one scale throughout (every 512 bytes of the bucket then hold a
// candidate, the worst case of the grid select); a call by itself, then a pair of compress and sum on eight streams (the
// grid select holds every SM through its shared steps, other calls' kernels run beside the list's):
//   float32  1M    0.2  39 / 37 | 34 / 36      20 / 29 | 20 / 29
//            3M    0.2  51 / 44 | 46 / 43      34 / 42 | 30 / 42
//            6.5M  0.13 57 / 60 | 55 / 61      47 / 55 | 45 / 58      0.2  72 / 62 | 69 / 63      59 / 62 | 55 / 62
//            16M   0.13 84 / 75 | 81 / 98      89 / 93 | 87 / 120     0.15 100 / 78 | 95 / 99     99 / 95 | 94 / 123
//            40M   0.13 172 / 135 | 172 / 186  200 / 180 | 195 / 240  0.2  232 / 149 | 205 / 193  268 / 204 | 248 / 249
//   bfloat16 3M    0.2  46 / 41 | 43 / 40      29 / 38 | 28 / 39
//            12M   0.1  61 / 57 | 58 / 63      53 / 65 | 53 / 70      0.15 65 / 59 | 65 / 67      63 / 69 | 67 / 75
//            34M   0.1  94 / 86 | 95 / 112     116 / 114 | 112 / 151  0.15 125 / 95 | 131 / 123   148 / 127 | 147 / 163
//            67M   0.1  161 / 135 | 165 / 188  211 / 192 | 212 / 253  0.15 212 / 147 | 225 / 208  276 / 216 | 278 / 277
//   with a residual, which the list stage subtracts from by scattered reads and writes (one call by itself):
//   float32  6.5M  0.125 63 / 67 | 61 / 68    0.15 64 / 67 | 61 / 67     0.2  81 / 68 | 79 / 67
//            16M   0.125 115 / 101 | 117 / 104  25M 168 / 146 | 164 / 159  45M 275 / 240 | 274 / 256
//   bfloat16 6.5M  0.125 63 / 63 | 60 / 63    16M 112 / 97 | 110 / 101   45M 249 / 223 | 253 / 241
// For a call by itself the lines are where several scales gain a fifth and one scale loses less than that; below 4M
// elements, where a call gains a tenth and calls on streams lose a quarter, the list keeps what it is made for (a quarter).
// many_calls (nsml_set_list_block_candidates above its default, the list stage then has fewer blocks): the list up to a
// quarter, but for large buckets, where from 0.2 on both kinds of data gain (40M float32 275 / 194 | 254 / 246, 34M bfloat16
// 178 / 140 | 189 / 177; 20M 108 / 110 | 111 / 134).
template <int VT>  // element type of what is selected from
inline double dense_from(int64_t n, bool many_calls = false, bool residual = false) {
  if (many_calls) return n < 32000000 ? 0.25 : 0.2;
  if (n < 4000000) return 0.25;
  if (n < 12000000) return 0.2;
  if (n < 40000000 && !residual) return 0.15;
  return VT == NSML_F32 ? 0.125 : 0.1;
}

// What k_select_grid is launched with.  grid = 0: it does not take the call.
struct GridPlan {
  unsigned int grid = 0, segs = 0, rows = 0, cap = 0, room = 0, rank_lo = 0, rank_hi = 0;
  size_t smem = 0;
  bool large = false;  // tables and lists lie in the workspace
};
// a block's tables in the workspace
template <int VT>
NSML_HD inline size_t grid_table_bytes(unsigned int rows) { return align_up(rows * grid_row_bytes<VT>(), 16); }

// VT: element type of what is selected from (float32 where a residual is added); grad_dtype: of the bucket; blocks: those
// that are resident at once, an even number; many_calls, residual: of dense_from.  The one place that decides: every size is taken,
// in a form that fits.
template <int VT>
inline GridPlan grid_plan(int64_t n, int64_t k, int grad_dtype, unsigned int blocks, bool many_calls = false,
                          bool residual = false) {
  GridPlan g;
  if ((double)k < dense_from<VT>(n, many_calls, residual) * (double)n) return g;
  // Bounds four standard deviations either side of the threshold's expected rank: one call in 16,000 takes another round
  // (3 us), the others have a window a third narrower than with six.
  const SamplePlan plan = sample_plan(n, k, grad_dtype, 4.0);
  const double keys = sampled_keys(grad_dtype);
  g.rank_lo = plan.rank_lo == 0 && k != n ? (unsigned int)keys + 1 : plan.rank_lo;  // (nearly everything is kept: an upper bound alone)
  g.rank_hi = plan.rank_hi;
  g.segs = (unsigned int)(((unsigned long long)n + grid_seg<VT>() - 1) / grid_seg<VT>());
  const unsigned int grid = g.segs < blocks ? g.segs : blocks;
  g.rows = (g.segs + grid - 1) / grid;
  // room for twice the keys that are to be expected inside the window, the rest of the shared memory for slices
  const double window = g.rank_lo == 0 ? 0.05 : (double)(g.rank_lo - g.rank_hi) / keys;
  const double entries = window * (double)n / ((double)grid * kGridWarps), twice = entries * 2.0 + 64.0;
  g.cap = twice < (double)kGridMaxCap ? (unsigned int)twice / 8 * 8 : kGridMaxCap;
  // Large buckets, whose tables (or places in the lists, 16 bits) do not fit, or whose lists would overflow (every phase then
  // walks all slices again), have both in the workspace: the tables, 0.14 bytes an element, in the place of the candidate
  // list's offsets, the lists, eight bytes an entry, in that of its values and of the raw values.  us, in shared memory / in
  // the workspace, by the entries a warp is to expect (there is room for 384): 64M float32 at 0.5 (216) 306 / 407, 100M at
  // 0.2 (264) 505 / 541, 100M at 0.5 (337) 631 / 589, 120M at 0.5 (405) 824 / 736, 150M at 0.2 (411) 977 / 801; bfloat16 at
  // 0.2 134M (254) 228 / 287, 270M (509) 568 / 516.
  g.large = g.rows > grid_max_rows<VT>() || grid_smem<VT>(g.rows, g.cap, 0) > kGridSmem || entries * kGridListMargin > (double)kGridMaxCap;
  if (g.large) {
    const double most = (double)n / ((double)grid * kGridWarps);
    g.cap = (unsigned int)(twice < most ? twice : most) / 8 * 8;
  }
  const size_t fixed = g.large ? grid_smem<VT>(0, 0, 0) : grid_smem<VT>(g.rows, g.cap, 0);
  const size_t room = (kGridSmem - fixed) / kGridSliceBytes, slices = (size_t)g.rows * kGridWarps;
  g.room = (unsigned int)(room < slices ? room : slices);
  g.smem = fixed + (size_t)g.room * kGridSliceBytes;
  g.grid = grid;
  return g;
}

}  // namespace nsml
