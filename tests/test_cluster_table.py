"""The table that keeps the runtime's answers on clusters (ClusterTable in
dlm_internal.h), compiled for the host with stand-ins for the query."""
import os
import shutil
import subprocess

import pytest

from paper_2608_02625_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "dlm_internal.h"

#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }

int main() {
  static dlm::ClusterTable table;
  int kernel = 0, other = 0, asked = 0;
  auto answer = [&](int n) { return [&asked, n] { ++asked; return n; }; };
  // a failed query is not kept
  CHECK(table.get({&kernel, 0, 8, 256, 0}, answer(-1)) == 0 && asked == 1);
  CHECK(table.get({&kernel, 0, 8, 256, 0}, answer(18)) == 18 && asked == 2);
  CHECK(table.get({&kernel, 0, 8, 256, 0}, answer(-1)) == 18 && asked == 2);
  // none at all is an answer
  CHECK(table.get({&kernel, 0, 16, 256, 0}, answer(0)) == 0 && asked == 3);
  CHECK(table.get({&kernel, 0, 16, 256, 0}, answer(5)) == 0 && asked == 3);
  // every part of the key counts
  CHECK(table.get({&other, 0, 8, 256, 0}, answer(1)) == 1);
  CHECK(table.get({&kernel, 1, 8, 256, 0}, answer(2)) == 2);
  CHECK(table.get({&kernel, 0, 4, 256, 0}, answer(3)) == 3);
  CHECK(table.get({&kernel, 0, 8, 128, 0}, answer(4)) == 4);
  CHECK(table.get({&kernel, 0, 8, 256, 64}, answer(6)) == 6);
  CHECK(table.get({&kernel, 0, 8, 256, 0}, answer(9)) == 18 && asked == 8);
  // a full table asks each time
  for (int i = 0; i < 300; ++i) CHECK(table.get({&kernel, 2, i, 256, 0}, answer(i)) == i);
  const int before = asked;
  CHECK(table.get({&kernel, 2, 299, 256, 0}, answer(7)) == 7 && asked == before + 1);
  CHECK(table.get({&kernel, 0, 8, 256, 0}, answer(9)) == 18 && asked == before + 1);
  return 0;
}
"""


def test_answers_are_kept_by_their_whole_key_and_failures_are_not(tmp_path):
    if not shutil.which("nvcc") and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    src, exe = str(tmp_path / "table.cu"), str(tmp_path / "table")
    with open(src, "w") as f:
        f.write(PROGRAM)
    r = subprocess.run([build.nvcc(), "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC] + build.ARCH + [src, "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
