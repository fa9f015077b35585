"""The rule that gives a trace of start columns its end column, compiled for
the host: whatever a batch's results hold after a device wait gave up (columns
of an earlier, longer reference, memory never written), no trace reads beyond
the reference image or runs for more steps than a sweep."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
SOURCE = r"""
#include <cstdio>
#include "haru_internal.h"
using namespace haru;
int main() {
  const int64_t cols[] = {INT64_MIN, -2, -1, 0, 1, 510, 2047, 2048, 59795, 59796, 1ll << 31, (1ll << 31) + 7,
                          1ll << 40, INT64_MAX};
  const long refs[] = {1, 2048, 59796, 1l << 31};
  int bad = 0;
  for (long N : refs)
    for (int64_t col : cols)
      for (int gave_up = 0; gave_up < 2; ++gave_up) {
        const long end = trace_end(col, N, gave_up);
        const bool traced = !gave_up && col >= 0 && col < N;
        bad += end != (traced ? static_cast<long>(col) : -1);
        for (int S = 1; S <= kMaxS; ++S) {
          if (end < 0) continue;
          const long t_end = (end + 32l * S - 1 + kChunk) / kChunk * kChunk;
          bad += t_end > sweep_steps(S, N) || t_end - 1 >= N + kRefPad;
        }
      }
  std::printf("%d\n", bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs the CUDA compiler")
def test_trace_end_stays_on_the_reference(tmp_path):
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(SOURCE)
    subprocess.check_call([NVCC, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                           os.path.join(ROOT, "paper_2211_07340_gb300", "csrc"), str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"
