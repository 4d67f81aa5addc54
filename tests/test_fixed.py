"""The fixed-point functions of csrc/fixed.cuh on the host against long double: sine and cosine,
logarithm and exponential within the bounds that the header states, and the product of the FP64
likelihood's sums against 128-bit integers, with every extreme of the halves."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2410_05190_gb300", "csrc")

PROGRAM = r"""
#include "fixed.cuh"
#include <cmath>
#include <cstdio>
#include <algorithm>
using namespace mbis;
typedef long double real;
static uint64_t s = 88172645463325252ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static const real kPiL = 3.14159265358979323846264338327950288L;

static void turns(uint64_t P, int64_t& co, int64_t& si) {
  const TrigCell c = trig_cell(P);
  trig_eval(c, pair32(kTrigTable[c.i][0]), pair32(kTrigTable[c.i][1]), co, si);
}

static double trig() {
  real worst = 0;
  auto one = [&](uint64_t P) {
    int64_t co, si;
    turns(P, co, si);
    const real a = (real)(int64_t)P * (kPiL * 0x1p-63L);
    worst = std::max(worst, std::fabs((real)co * 0x1p-62L - std::cos(a)));
    worst = std::max(worst, std::fabs((real)si * 0x1p-62L - std::sin(a)));
  };
  for (int i = 0; i < 2000000; ++i) one(rnd());
  for (uint64_t i = 0; i < 256; ++i)  // the cells' edges and centres
    for (int d = -2; d <= 2; ++d) one((i << 56) + (uint64_t)d);
  return (double)(worst / 2.7e-17L);
}

static double logarithm() {
  real worst = 0;
  auto one = [&](uint64_t m) {
    const int64_t* e = kLogTable[log_cell(m)];
    worst = std::max(worst, std::fabs((real)log_frac(m, (uint32_t)e[0], e[1]) * 0x1p-62L - std::log((real)m * 0x1p-63L)));
  };
  for (int i = 0; i < 1000000; ++i) one(rnd() | (1ull << 63));
  for (uint64_t i = 128; i < 256; ++i) { one(i << 56); one((i << 56) | 0xffffffffffffffull); }
  return (double)(worst / (8 * 0x1p-62L));
}

static double exponential() {
  real worst = 0;
  auto one = [&](double d) {
    int32_t n;
    uint64_t t;
    const int32_t j = exp_cell(d, n, t);
    const double got = exp_eval(n, t, kExpTable[j]);
    const real want = std::exp((real)d);
    const real ulp = (real)(std::nextafter((double)want, 2.0) - (double)want);
    worst = std::max(worst, std::fabs((real)got - want) / ulp);
  };
  for (int i = 0; i < 1000000; ++i) {
    const double u = (double)(rnd() >> 11) * 0x1p-53;
    one(-700.0 * u);
    one(-std::exp(-40.0 * u) * 0.7);
  }
  for (int k = 0; k <= 1000; ++k) { one(-0.69314718055994530942 * k); one(-0.7 * k); }
  one(0.0);
  one(-0.0);
  one(-5e-324);
  return (double)(worst / 0.8L);
}

// sums of a data value times e^(-i phi): unit 2^-120 products, kept by their high words
static double product() {
  const int32_t low[] = {INT32_MIN, INT32_MIN + 1, -1, 0, 1, INT32_MAX};
  double worst = 0;
  for (int i = 0; i < 1000000; ++i) {
    int64_t co, si;
    turns(i % 8 ? rnd() : (uint64_t)i << 60, co, si);
    int64_t w[2];
    for (int64_t& x : w) {
      x = (int64_t)rnd() >> (5 + rnd() % 30);  // below 2^58
      if (rnd() & 1) x = (x & ~0xffffffffll) + low[rnd() % 6];
    }
    int64_t ar = 0, ai = 0;
    add_rotated(pair32(w[0]), pair32(w[1]), pair32(co), pair32(si), ar, ai);
    const __int128 er = (__int128)w[0] * co + (__int128)w[1] * si, ei = (__int128)w[1] * co - (__int128)w[0] * si;
    worst = std::max(worst, std::fabs((double)(((__int128)ar << 64) - er) * 0x1p-64));
    worst = std::max(worst, std::fabs((double)(((__int128)ai << 64) - ei) * 0x1p-64));
  }
  return worst / 2.0;  // two dropped products of low halves (a quarter each) and one truncation
}

int main() {
  for (const auto& e : kTrigTable)  // trig_eval negates the halves of the sine
    if (pair32(e[1]).l == INT32_MIN) return 1;
  std::printf("%g %g %g %g\n", trig(), logarithm(), exponential(), product());
  return 0;
}
"""


@pytest.mark.parametrize("opt", ["-O0", "-O2"])
def test_fixed_point_functions_keep_their_bounds(tmp_path, opt):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", opt, "-std=c++17", "-I", CSRC, "-x", "c++", str(src), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    fractions = dict(zip(["sine and cosine", "logarithm", "exponential", "product"],
                         map(float, out.stdout.split())))  # of each bound
    assert all(v <= 1.0 for v in fractions.values()), fractions
