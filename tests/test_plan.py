"""Whether the grid select takes a call, and what it is then launched with (nsml_plan.h), over every size: the host code is
compiled here and asked, no GPU needed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "nsml_plan.h"
using namespace nsml;

static long taken = 0, left = 0, large = 0, wrong = 0;

// what the kernel relies on, beside that the driver accepts the launch
template <int VT>
static void check(int64_t n, double ratio, int grad_dtype, unsigned int blocks, bool many_calls, bool residual = false) {
  int64_t k = (int64_t)std::ceil(ratio * (double)n);
  if (k > n) k = n;
  const GridPlan g = grid_plan<VT>(n, k, grad_dtype, blocks, many_calls, residual);
  if (g.grid == 0) {  // less is kept
    wrong += (double)k >= dense_from<VT>(n, many_calls, residual) * (double)n;
    ++left;
    return;
  }
  ++taken;
  const uint64_t seg = grid_seg<VT>();
  bool ok = g.smem <= kGridSmem && g.smem == grid_smem<VT>(g.large ? 0 : g.rows, g.large ? 0 : g.cap, g.room);
  ok &= g.grid <= blocks && (g.grid % 2 == 0 || g.rows == 1);
  ok &= (uint64_t)g.segs * seg >= (uint64_t)n && (uint64_t)(g.segs - 1) * seg < (uint64_t)n;
  ok &= (uint64_t)g.rows * g.grid >= g.segs && g.rows >= 1;
  ok &= (uint64_t)g.rows * g.grid * seg < (1ull << 32);               // element indices of any row
  if (g.large) {                                                      // in the workspace: 2 bytes an element, 4 and 4
    ok &= (uint64_t)g.grid * grid_table_bytes<VT>(g.rows) <= 2ull * n;
    ok &= (uint64_t)g.grid * kGridWarps * g.cap <= (uint64_t)n;
  } else {
    ok &= g.rows <= grid_max_rows<VT>();                              // an entry's place in 16 bits
    ok &= g.cap <= kGridMaxCap;
  }
  ok &= g.room <= g.rows * kGridWarps && g.room < 0xFFFFu;            // a slice's place + 1 in 16 bits, 0xFFFF apart
  ok &= (g.rank_lo == 0) == (k == n) && (g.rank_lo == 0 || g.rank_hi < g.rank_lo);
  large += g.large;
  if (!ok && wrong++ < 10)
    std::printf("n %lld ratio %g type %d of %d blocks %u: grid %u segs %u rows %u cap %u room %u smem %zu ranks %u %u\n", (long long)n, ratio, VT,
                grad_dtype, blocks, g.grid, g.segs, g.rows, g.cap, g.room, g.smem, g.rank_lo, g.rank_hi);
}

int main() {
  for (unsigned int blocks : {148u, 132u, 80u, 192u}) {
    std::vector<int64_t> at;
    for (int64_t rows = 1; rows <= 4096; ++rows)  // around every number of rows, of either type
      for (int64_t seg : {4096, 8192})
        for (int64_t d : {-1, 0, 1}) at.push_back(rows * blocks * seg + d);
    for (double x = 163841; x < 2.2e9; x *= 1.01) at.push_back((int64_t)x);
    at.push_back(163841);
    at.push_back(NSML_MAX_N);
    for (int64_t n : at) {
      if (n <= 163840 || n > NSML_MAX_N) continue;
      for (double ratio : {0.05, 0.1, 0.125, 0.13, 0.2, 0.3, 0.5, 0.9, 0.999, 0.99999, 1.0}) {
        for (bool many_calls : {false, true}) {
          check<NSML_F32>(n, ratio, NSML_F32, blocks, many_calls);
          check<NSML_F32>(n, ratio, NSML_F32, blocks, many_calls, true);
          check<NSML_F32>(n, ratio, NSML_BF16, blocks, many_calls, true);
          check<NSML_BF16>(n, ratio, NSML_BF16, blocks, many_calls);
        }
      }
    }
  }
  std::printf("%ld taken, %ld of them large, %ld left, %ld wrong\n", taken, large, left, wrong);
  return wrong == 0 && taken > large && large > 0 && left > 0 ? 0 : 1;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_every_call_that_is_taken_fits(tmp_path):
    source, binary = tmp_path / "plan.cpp", tmp_path / "plan"
    source.write_text(PROGRAM)
    flags = ["-std=c++17", "-O1", "-Wall", "-Werror", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2506_16235_b200", "csrc")]
    subprocess.run(["g++", *flags, str(source), "-o", str(binary)], check=True, timeout=120)
    got = subprocess.run([str(binary)], capture_output=True, text=True, timeout=120)
    assert got.returncode == 0, got.stdout
