"""The kernels' multiply-high division (FastDiv, posmod of kubo_internal.cuh), compiled for the host.

A quotient by the rounded-up reciprocal alone is exact only while a d < 2^32; the row split of the
Fourier coefficients (65,536 rows of up to 2,500 pairs) and the phases of long mesh axes (j R mod N) go past that.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstdio>
#include "kubo_internal.cuh"
using namespace kubo;
static bool bad(uint32_t a, uint32_t d) {
  uint32_t r;
  const uint32_t q = FastDiv(d).divmod(a, r);
  if (q == a / d && r == a % d) return false;
  std::printf("divmod %u %u -> %u %u\n", a, d, q, r);
  return true;
}
int main() {
  // (row, pair) of every index near a row's end, over the padded pair counts of up to 5,000 lattice vectors
  for (uint32_t d = 32; d <= 2528; d += 32)
    for (uint64_t m = 1; m * d < (1ull << 32) && m <= 600000; m += 1 + m / 4096)
      for (int o = -3; o < 2; ++o)
        if (bad((uint32_t)(m * d + o), d)) return 1;
  // the ends of the range, for divisors of every size
  for (uint64_t d = 1; d < (1ull << 31); d += 1 + d / 97)
    for (uint32_t back = 0; back < 3; ++back)
      for (uint32_t a : {0xFFFFFFFFu - back, (uint32_t)(0xFFFFFFFFull / d * d - 1 + back), (uint32_t)d - 1u + back})
        if (bad(a, (uint32_t)d)) return 1;
  // mesh phases j R mod N: long axes, far lattice vectors, both signs
  for (int N : {1, 2, 3, 64, 9973, 65536, 65537, 90001, 1000003, 2147483647})
    for (int r : {0, 1, -1, 5, -7, 1000, -65537, 2147483647})
      for (int j = N - 1; j >= 0 && j > N - 40; --j) {
        const long long x = (long long)j * r, want = ((x % N) + N) % N;
        if (posmod(x, FastDiv((uint32_t)N)) != want) { std::printf("posmod %lld %d\n", x, N); return 1; }
      }
  std::puts("ok");
  return 0;
}
"""


def test_division_is_exact_over_the_whole_range(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "fastdiv.cu", tmp_path / "fastdiv"
    src.write_text(SRC)
    inc = [f"-I{ROOT}/include", f"-I{ROOT}/paper_2309_06675_gb300/csrc"]
    subprocess.run([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a"] + inc +
                   [str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
