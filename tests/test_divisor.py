"""Division by a partition's layer size and head count as a multiplication (Divisor), on the CPU: every
quotient's first and last dividend below 2^31 that matter, for small, large and power-of-two divisors."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "kvtier_internal.cuh"
static uint32_t by(const kvt::Divisor& d, uint32_t x) { return d.mul ? (uint32_t)((uint64_t)x * d.mul >> 32) >> d.shift : x; }
int main() {
  std::mt19937_64 r(1);
  const uint32_t top = 0x7FFFFFFFu;
  for (int i = 0; i < 200000; ++i) {
    uint32_t d = i < 4096 ? (uint32_t)i + 1u : (uint32_t)(r() >> (33 + r() % 31)) + 1u;
    if (i % 7 == 0) d = (1u << r() % 31) + (uint32_t)(r() % 3) - 1u;
    if (d == 0u || d > top) continue;
    const kvt::Divisor v(d);
    const uint32_t q = (uint32_t)(r() >> 33) / d;
    for (uint32_t x : {0u, d - 1u, d, q * d, q * d + d - 1u, top / d * d, top / d * d - 1u, top})
      if (x <= top && by(v, x) != x / d) { std::printf("%u / %u gives %u\n", x, d, by(v, x)); return 1; }
  }
  return 0;
}
"""


def test_quotients(tmp_path):
    src, exe = tmp_path / "divisor.cu", tmp_path / "divisor"
    src.write_text(PROGRAM)
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-std=c++17", "-O1", "-gencode",
                    "arch=compute_100a,code=sm_100a", "-diag-suppress", "186", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2604_26968_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
