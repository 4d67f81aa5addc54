"""The integer-pipe conversions of csrc/fpcvt.cuh against the language's on the host, bit for
bit: random bit patterns, every exponent's edges, ties, carries, zeros, subnormals, infinities
and NaN."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2410_05190_gb300", "csrc")

PROGRAM = r"""
#include "fpcvt.cuh"
#include <cmath>
#include <cstdio>
using namespace mbis;
static uint64_t s = 88172645463325252ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static long bad = 0;
static void check(uint64_t b) {
  const double x = double_of((uint32_t)(b >> 32), (uint32_t)b);
  const float want = (float)x, got = to_float(x);
  float h, l;
  split_float(x, h, l);
  const float wl = (float)(x - (double)want);
  auto same = [](float p, float q) { return bits_of(p) == bits_of(q) || (std::isnan(p) && std::isnan(q)); };
  bad += !same(want, got) + !same(want, h) + !same(wl, l);
  bad += is_positive(x) != (x > 0.0);
  bad += is_below_one(x) != (std::fabs(x) < 1.0);
  bad += is_below_exp2(x, 20) != (std::fabs(x) < 1048576.0);
  bad += is_finite(x) != std::isfinite(x);
}
static void check32(uint32_t b) {
  const float f = float_of(b);
  uint32_t h0, l0, h1, l1;
  words_of((double)f, h0, l0);
  words_of(to_double(f), h1, l1);
  if (!std::isnan(f)) bad += h0 != h1 || l0 != l1; else bad += !std::isnan(to_double(f));
  words_of((double)(int32_t)b, h0, l0);
  words_of(to_double((int32_t)b), h1, l1);
  bad += h0 != h1 || l0 != l1;
}
int main() {
  const uint64_t edge[] = {0, 1, 0x0fffffff, 0x10000000, 0x10000001, 0x1fffffff, 0x20000000, 0x2fffffff, 0x30000000,
                           0x30000001, 0x3fffffff, 0xfffffffffffffull, 0xfffffe0000000ull, 0xfffffefffffffull,
                           0xffffff0000000ull, 0xffffff0000001ull};
  for (uint64_t e = 0; e < 2048; ++e)
    for (uint64_t m : edge)
      for (uint64_t sg = 0; sg < 2; ++sg) check(sg << 63 | e << 52 | m);
  for (long i = 0; i < 4000000; ++i) {
    check(rnd());
    check((rnd() & 0x800fffffffffffffull) | (880 + rnd() % 290) << 52);  // the FP32 range
    check((rnd() & 0x800fffffe0000000ull) | (940 + rnd() % 215) << 52 | 0x10000000);  // ties
  }
  for (uint64_t b = 0; b < (1ull << 32); b += 331) check32((uint32_t)b);
  const uint32_t f[] = {0, 0x80000000u, 1, 0x007fffff, 0x00800000, 0x7f7fffff, 0x7f800000, 0xff800000u, 0x7fc00000,
                        0x00ffffff, 0x01000000, 0x01000001, 0xff000000u, 0xfeffffffu, 0xff000001u};
  for (uint32_t b : f) check32(b);
  std::printf("%ld\n", bad);
  return bad != 0;
}
"""


@pytest.mark.parametrize("opt", ["-O0", "-O2"])
def test_integer_conversions_are_the_languages(tmp_path, opt):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", opt, "-std=c++17", "-I", CSRC, "-x", "c++", str(src), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "0", out.stdout
