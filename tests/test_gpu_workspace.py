"""Workspace sizing through the library's own C++ functions, from a small
program that is compiled and linked against it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not os.path.exists(NVCC), reason="needs the CUDA compiler")]


def run(tmp_path, body):
    import paper_2211_07340_gb300 as haru
    lib = os.path.dirname(haru.build_library())
    src, exe = tmp_path / "sizes.cu", tmp_path / "sizes"
    src.write_text("#include <cstdio>\n#include \"engine.h\"\nusing namespace haru;\nint main() {\n" + body + "\n}\n")
    subprocess.check_call([NVCC, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                           os.path.join(ROOT, "paper_2211_07340_gb300", "csrc"), str(src), "-o", str(exe), "-L", lib,
                           "-lharu", "-Xlinker", "-rpath=" + lib])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


# references below and above the line of traced start columns
@pytest.mark.parametrize("n", [1000, 59796])
def test_reserve_upto_covers_every_smaller_batch(tmp_path, n):
    """After ws_reserve_upto(300) no batch of 1..300 queries allocates, in any form."""
    out = run(tmp_path, """
  LaunchCfg lc;
  lc.sms = 152;
  lc.N = %d;
  for (int prec : {HARU_FP32, HARU_INT16, HARU_INT16_ACC32, kPrecF32Span, kPrecWideSpan}) {
    Workspace ws;
    if (ws_reserve_upto(ws, prec, 300, lc) != cudaSuccess) return 1;
    auto caps = [&] {
      return std::vector<size_t>{ws.cap_groups, ws.cap_done, ws.cap_items, ws.cap_states, ws.cap_bests,
                                 ws.cap_checkpoints, ws.cap_qstats, reinterpret_cast<size_t>(ws.states),
                                 reinterpret_cast<size_t>(ws.checkpoints), reinterpret_cast<size_t>(ws.bests)};
    };
    const auto before = caps();
    int grew = 0;
    for (uint32_t q = 1; q <= 300; ++q) {
      if (ws_reserve(ws, prec, q, lc) != cudaSuccess) return 1;
      grew += caps() != before;
    }
    std::printf("%%d ", grew);
    ws_free(ws);
  }
  return 0;""" % n)
    assert out.split() == ["0"] * 5


# (precision, device bytes a query at most: what a batch of this size took before the static schedule, whose third
# segment must not cost a caller at the memory's end the batch)
@pytest.mark.parametrize("prec,most", [("HARU_FP32", 22_800), ("HARU_INT16", 11_500)])
def test_memory_of_very_large_batches(tmp_path, prec, most):
    nq = 1 << 20
    out = run(tmp_path, """
  LaunchCfg lc;
  lc.sms = 152;
  lc.N = 59796;
  Workspace ws;
  size_t before, after, all;
  cudaFree(nullptr);
  cudaMemGetInfo(&before, &all);
  if (ws_reserve(ws, %s, %du, lc) != cudaSuccess) return 1;
  cudaMemGetInfo(&after, &all);
  std::printf("%%zu", before - after);
  ws_free(ws);
  return 0;""" % (prec, nq))
    assert int(out) <= nq * most


def test_checkpoints_of_very_large_batches(tmp_path):
    """Beside 20.3 KB of other buffers an item (above) 4 checkpoints of 4 KB stay below the 39,100 bytes a start-column
    query took before there were any."""
    out = run(tmp_path, """
  std::printf("%d %d", checkpoint_cap((1u << 22) - 1, 59796), checkpoint_cap(1u << 22, 59796));
  return 0;""")
    assert out.split() == ["8", "4"]
