"""Which four events the event reduction takes for entries in a row (is_run), on the CPU: for ids around 0,
around the pool's end and around 2^32, where sums wrap, and pools of every remainder modulo 4, a vector is a
run only if its ids follow each other as whole numbers and everything that a run reads lies inside the pool."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "kv_score_device.cuh"
template <bool PACKED> bool wrong(uint32_t n, uint32_t start, uint32_t last_step) {
  const uint32_t id[4] = {start, start + 1u, start + 2u, start + last_step};
  // a run reads the words of four pair bytes that hold its first and its last entry
  const unsigned long long end = ((unsigned long long)start + 3u) / 4u * 4u + 4u;
  const bool want = last_step == 3u && (PACKED || start % 4u == 0u) && end <= n;
  if (kvt::is_run(id, n, PACKED) == want) return false;
  std::printf("packed %d, pool of %u, start %u, last step %u: %d\n", (int)PACKED, n, start, last_step, (int)!want);
  return true;
}
int main() {
  int bad = 0;
  const uint32_t pools[] = {1, 2, 3, 4, 5, 6, 7, 8, 9, 4096, 11133, 11134, 11135, 11136, 0x7FFFFFFC, 0x7FFFFFFD, 0x7FFFFFFE, 0x7FFFFFFF};
  for (uint32_t n : pools)
    for (uint32_t from : {0u, n})
      for (int d = -12; d <= 12; ++d)
        for (uint32_t last_step : {3u, 4u, 2u})
          bad += wrong<true>(n, from + (uint32_t)d, last_step) + wrong<false>(n, from + (uint32_t)d, last_step);
  return bad != 0;
}
"""


def test_runs(tmp_path):
    src, exe = tmp_path / "runs.cu", tmp_path / "runs"
    src.write_text(PROGRAM)
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-std=c++17", "-O1", "-gencode",
                    "arch=compute_100a,code=sm_100a", "-diag-suppress", "186", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2604_26968_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
