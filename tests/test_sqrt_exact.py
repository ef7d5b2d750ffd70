"""The integer-pipe square root (mcx::sqrt_rn) and the truncating fp32 view of
a double against the host's IEEE arithmetic, from the header itself: uniform
arguments 1 - s, every exponent of the direction sampler's range, and the
neighbours of exact squares, where the rounding is closest to a tie."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_06362_gb300", "csrc")

PROGRAM = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#define __constant__
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
static float __uint_as_float(uint32_t b) { float f; memcpy(&f, &b, 4); return f; }
#include "fp_exact.cuh"
static double of(uint64_t b) { double x; memcpy(&x, &b, 8); return x; }
int main() {
  std::mt19937_64 r(1);
  long bad = 0;
  for (long i = 0; i < 3000000; ++i) {
    double x;
    if (MODE == 0) x = 1.0 - (double)(r() >> 11) * 0x1p-53;
    else if (MODE == 1) x = of((r() & ((1ull << 52) - 1)) | ((uint64_t)(1023 - (int)(r() % 60)) << 52));
    else {
      const double y = (double)((1u << 26) + (uint32_t)(r() % (1u << 26))) * 0x1p-27;
      const double s = y * y;
      uint64_t b; memcpy(&b, &s, 8);
      x = of(b + r() % 5 - 2);
    }
    const double got = mcx::sqrt_rn(x), want = std::sqrt(x);
    const float t = mcx::f32_trunc(x);
    if (memcmp(&got, &want, 8) || !mcx::f32_range(x) || !(t <= x) || !(x - t < x * 0x1p-23)) ++bad;
  }
  printf("%ld\n", bad);
}
"""


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_sqrt_and_fp32_view(tmp_path, mode):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-DMODE=%d" % mode, "-I", CSRC, str(src), "-o", exe],
                   check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout.strip() == "0"
