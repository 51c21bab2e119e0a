"""The attention masks' key ranges (key_ranges and all_rows_use in dlm_common.cuh,
mask_block in dlm_internal.h), compiled for the host and compared with the masks'
definition key by key."""
import os
import shutil
import subprocess

import pytest

from paper_2608_02625_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "dlm_common.cuh"
#include "dlm_internal.h"

static bool allowed(int mode, long long block, int row, int key, int p) {
  if (key < p) return true;
  if (row < p) return false;
  const long long own = (row - p) / block, other = (key - p) / block;
  return mode == DLM_ATTN_BLOCK_CAUSAL ? other <= own : other == own;
}

static int ranges() {
  const int blocks[] = {1, 7, 64, 100, 1000, 0x7FFFFFFF - 70, 0x7FFFFFFF};  // p + block overflows for the last two
  for (int mode = 1; mode <= 2; ++mode)
    for (int block : blocks)
      for (int n = 1; n <= 140; n += 3)
        for (int p = 0; p <= n; p += 9)
          for (int row = 0; row < n; ++row) {
            const dlm::KeyRanges r = dlm::key_ranges(mode, dlm::mask_block(block, n), row, n, p);
            for (int key = 0; key < n; ++key)
              if ((key < r.hi1 || (key >= r.lo2 && key < r.hi2)) != allowed(mode, block, row, key, p)) {
                std::printf("mode %d block %d n %d p %d row %d key %d\n", mode, block, n, p, row, key);
                return 1;
              }
          }
  return 0;
}

// A tile may count as every row's only where each row may use each of its keys.
static int tiles() {
  const int blocks[] = {7, 20, 64, 100, 128, 1000, 0x7FFFFFFF}, heights[] = {1, 32, 64, 112, 128}, prompts[] = {0, 10, 20, 64, 100, 128};
  int whole = 0;
  for (int mode = 1; mode <= 2; ++mode)
    for (int block : blocks)
      for (int p : prompts)
        for (int n : {65, 128, 200, 333})
          for (int m : heights)
            for (int r0 = 0; p <= n && r0 < n; r0 += m) {
              const int r1 = (r0 + m < n ? r0 + m : n) - 1;
              const int blk = dlm::mask_block(block, n);
              const dlm::KeyRanges first = dlm::key_ranges(mode, blk, r0, n, p), last = dlm::key_ranges(mode, blk, r1, n, p);
              for (int key0 = 0; key0 < n; key0 += 64) {
                if (!dlm::all_rows_use(first, last, key0, key0 + 64)) continue;
                ++whole;
                for (int row = r0; row <= r1; ++row)
                  for (int key = key0; key < key0 + 64; ++key)
                    if (key >= n || !allowed(mode, block, row, key, p)) {
                      std::printf("mode %d block %d n %d p %d rows %d..%d keys %d..: row %d key %d\n", mode, block, n, p, r0, r1,
                                  key0, row, key);
                      return 1;
                    }
              }
            }
  return whole == 0;  // some tile is
}

int main(int argc, char** argv) {
  (void)argv;
  return argc > 1 ? tiles() : ranges();
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("nvcc") and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("ranges")
    src, exe = str(d / "ranges.cu"), str(d / "ranges")
    with open(src, "w") as f:
        f.write(PROGRAM)
    r = subprocess.run([build.nvcc(), "-std=c++17", "-O1", "-I", build.INCLUDE, "-I", build.CSRC] + build.ARCH +
                       [src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@pytest.mark.parametrize("what", [[], ["tiles"]], ids=["ranges", "tiles"])
def test_matches_the_masks(program, what):
    r = subprocess.run([program] + what, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout or r.stderr
