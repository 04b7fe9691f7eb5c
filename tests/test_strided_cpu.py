"""for_strided (csrc/common.cuh), the loop over a row's entries, at the int32 limit of the entry
positions: every position once and none beyond the end.  Compiled for the host."""
import os
import shutil
import subprocess

import pytest

from paper_2407_16144_gb300 import _build

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None and
                                not os.path.exists("/usr/local/cuda/bin/nvcc"),
                                reason="nvcc not available")

PROGRAM = r"""
#include <climits>
#include <cstdio>
#include <cstdlib>
#include "common.cuh"
int main() {
  const int ends[] = {0, 1, 1000, INT_MAX - 1, INT_MAX};
  for (int e : ends)
    for (int len : {0, 1, 31, 300, 1000})
      for (int step : {1, 4, 32, 256}) {
        const int b = e - len;
        if (b < 0) continue;
        long long seen = 0, sum = 0;
        for (int first = 0; first < step; ++first)
          rh::for_strided(b, e, first, step, [&](int p) {
            if (p < b || p >= e || seen > len) { std::printf("out of range\n"); std::exit(1); }
            ++seen;
            sum += p - b;
          });
        if (seen != len || sum != (long long)len * (len - 1) / 2) return 2;
      }
  return 0;
}
"""


def test_entries_up_to_the_int32_limit(tmp_path):
    src, exe = tmp_path / "strided.cu", tmp_path / "strided"
    src.write_text(PROGRAM)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
