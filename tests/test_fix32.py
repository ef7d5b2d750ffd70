"""A float track length to int64 fixed point of scale 2^32 (mcs::fix32_from_float
and its integer form for long tracks), from the source itself with the
directed roundings it names, against the exact integer rounding: random
lengths of every binade, and those whose last 16 bits round up to 2^16 and
have to carry into the word above (2^-16 - 2^-40 is the simplest)."""
import os
import re
import subprocess

import pytest

SLAB = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_06362_gb300", "csrc", "slab.cuh")

PROGRAM = r"""
#include <cfenv>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __noinline__
#define __forceinline__ inline
static uint32_t __float_as_uint(float f) { uint32_t b; memcpy(&b, &f, 4); return b; }
static float __fadd_rz(float a, float b) { volatile float x = a, y = b; fesetround(FE_TOWARDZERO); volatile float s = x + y; fesetround(FE_TONEAREST); return s; }
static float __fadd_rn(float a, float b) { volatile float x = a, y = b; volatile float s = x + y; return s; }
static float __fsub_rn(float a, float b) { return __fadd_rn(a, -b); }
static float __fmul_rn(float a, float b) { volatile float x = a, y = b; volatile float s = x * y; return s; }
@SOURCE@
static long bad;
static void look(float v) {
  if (fix32_from_float(v) != std::llrint((double)v * 4294967296.0)) { ++bad; printf("%a\n", (double)v); }
}
int main() {
  const float one = 1.0f - 0x1p-24f;  // 24 ones
  for (int e = -40; e < 24; ++e) { look(std::ldexp(one, e)); look(std::ldexp(1.0f, e)); look(std::ldexp(1.5f, e)); }
  look(0.0f); look(0x1p-16f - 0x1p-40f); look(4194304.0f); look(std::nextafter(4194304.0f, 0.0f)); look(1e-45f);
  for (int k = 1; k < 4000; ++k) look((float)k * (0x1p-16f - 0x1p-40f));
  std::mt19937 r(1);
  for (int e = -40; e < 28; ++e)
    for (int i = 0; i < 20000; ++i) look(std::ldexp((float)(0x800000u | (r() & 0x7fffffu)), e - 23));
  printf("%ld\n", bad);
}
"""


@pytest.mark.parametrize("optimise", ["-O0", "-O2"])
def test_equals_the_exact_rounding(tmp_path, optimise):
    text = open(SLAB).read()
    source = re.search(r"static __device__ __noinline__ long long fix32_any.*?\n}\n.*?fix32_from_float\(float v\) \{.*?\n}\n", text, re.S)
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM.replace("@SOURCE@", source.group(0)))
    exe = str(tmp_path / "t")
    subprocess.run(["g++", optimise, "-std=c++17", "-ffp-contract=off", "-frounding-math", str(src), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout.strip() == "0"
