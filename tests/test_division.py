"""The collision's division by the small integers of M M^T and N N^T against
the IEEE quotient, compiled for the host from the kernels' own header: the same
bits for every normal quotient, down to the smallest ones that a run from
exact rest passes through (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

from paper_1608_04118_gb300 import build as B

SOURCE = r"""
#include "ltne_node.cuh"
#include <cfloat>
#include <cstdio>
static uint64_t state = 88172645463325252ull;
static uint64_t next() {  // xorshift64
  state ^= state << 13; state ^= state >> 7; state ^= state << 17;
  return state;
}
template <int D, typename C> static long wrong(int e_lo, int e_hi, long n) {
  long bad = 0;
  for (long k = 0; k < n; ++k) {
    const C s = C(1) + std::ldexp(C(next() >> (64 - (sizeof(C) == 8 ? 52 : 23))),
                                  sizeof(C) == 8 ? -52 : -23);
    const C x = std::ldexp(next() & 1 ? s : -s, e_lo + (int)(next() % (uint64_t)(e_hi - e_lo)));
    volatile C d = C(D);
    const C q = x / d;
    if (std::fabs(q) < (sizeof(C) == 8 ? C(DBL_MIN) : C(FLT_MIN))) continue;
    if (ltne::div_small<D, C>(x) != q) ++bad;
  }
  return bad;
}
template <typename C> static long all(int lo, int hi, long n) {
  return wrong<5, C>(lo, hi, n) + wrong<6, C>(lo, hi, n) + wrong<9, C>(lo, hi, n) +
         wrong<12, C>(lo, hi, n) + wrong<20, C>(lo, hi, n) + wrong<36, C>(lo, hi, n);
}
int main() {
  std::printf("%ld %ld %ld %ld\n", all<double>(-1022, 1000, 200000), all<double>(-1022, -1010, 200000),
              all<float>(-126, 120, 200000), all<float>(-126, -110, 200000));
}
"""


def test_division_by_small_integers_is_correctly_rounded(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "div.cu", str(tmp_path / "div")
    src.write_text(SOURCE)
    subprocess.run([nvcc, *B.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr",
                    "-Xcompiler", "-ffp-contract=off", "-I", B.CSRC, str(src), "-o", exe], check=True)
    got = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert got == ["0"] * 4, "wrong quotients: FP64 all, FP64 smallest, FP32 all, FP32 smallest"
