"""The flight logarithm's host copy under the undefined behaviour sanitizer:
its table form runs for every argument, also for those whose value it does not
give (u below 2^-8, 1 - u below 2^-21), and has to be defined there too."""
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
#include "mc_log.cuh"
int main() {
  std::mt19937_64 r(1);
  const uint64_t all = 1ull << 53;
  long bad = 0;
  auto look = [&](uint64_t n) {
    const double want = n ? -std::log1p(-(double)n * 0x1p-53) : 0.0, got = mclog::neglog1m_n(n);
    if (!(std::fabs(got - want) <= 4e-16 * want)) ++bad;
  };
  for (uint64_t n = 0; n < 5000; ++n) { look(n); look(all - 1 - n); look((1ull << 45) - 2500 + n); look(all - (1ull << 32) - 2500 + n); }
  for (int e = 0; e < 53; ++e)
    for (int i = 0; i < 2000; ++i) { const uint64_t n = (1ull << e) + r() % (1ull << e); look(n); look(all - n); }
  printf("%ld\n", bad);
}
"""


@pytest.mark.parametrize("optimise", ["-O0", "-O2"])
def test_every_argument_is_defined(tmp_path, optimise):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    made = subprocess.run(["g++", optimise, "-std=c++17", "-ffp-contract=off", "-fsanitize=undefined",
                           "-fno-sanitize-recover=all", "-I", CSRC, str(src), "-o", exe], capture_output=True, text=True)
    if "ubsan" in made.stderr:
        pytest.skip("no sanitizer runtime")
    assert made.returncode == 0, made.stderr
    ran = subprocess.run([exe], capture_output=True, text=True)
    assert ran.returncode == 0 and ran.stdout.strip() == "0", ran.stdout + ran.stderr
