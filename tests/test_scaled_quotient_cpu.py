"""The FP32 quotients of the scaled matrix values (csrc/quotient.cuh, the code
that runs on the device) against the division in FP64: the same FP32 number
over all exponents, on both sides of the ones where it divides instead, except
that a divisor whose significand is all ones may give a neighbour's rounding."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "quotient.cuh"
#include <cstdint>
#include <cstdio>
#include <initializer_list>
#include <limits>

static uint64_t s = 88172645463325252ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s * 2685821657736338717ull; }
static double make(uint64_t mant, int e, bool neg) {  // 1.mant 2^(e - 1023)
  uint64_t b = (uint64_t)neg << 63 | (uint64_t)e << 52 | (mant & ((1ull << 52) - 1));
  double d;
  std::memcpy(&d, &b, 8);
  return d;
}
static uint32_t bits(float f) { uint32_t b; std::memcpy(&b, &f, 4); return b; }

int main() {
  const int limits[] = {0, 1, 622, 623, 624, 1022, 1023, 1024, 1422, 1423, 1424, 2046, 2047};
  const uint64_t ones = (1ull << 52) - 1;
  long long bad = 0, neighbours = 0, done = 0;
  auto check = [&](double a, double c, bool exact) {
    const float got = ld::scaled_quotient(a, c, ld::quotient_reciprocal(c)), want = (float)(a / c);
    ++done;
    if (bits(got) == bits(want) || (got != got && want != want)) return;
    if (!exact && got == std::nextafter(want, got)) ++neighbours;
    else if (++bad < 10) std::printf("a %a c %a got %a want %a\n", a, c, got, want);
  };
  for (int k = 0; k < 3000000; ++k) {
    const uint64_t r = rnd();
    // Divisors over the reciprocal's range (2^-333 .. 2^333) and past it.
    const int ec = k % 7 == 0 ? 1 + (int)(r % 2046) : 1023 - 340 + (int)(r % 681);
    const int ea = k % 3 == 0 ? limits[(r >> 20) % 13]
                 : k % 3 == 1 ? (int)((r >> 20) % 2048)
                              : ec - 130 + (int)((r >> 20) % 261);  // FP32-sized quotients
    if (ea < 0 || ea > 2047) continue;
    const uint64_t mc = k % 11 == 0 ? ones : k % 13 == 0 ? 0 : rnd();
    const double c = make(mc, ec, k % 17 == 0);
    check(make(k % 5 == 0 ? rnd() & ~((1ull << 28) - 1) : rnd(), ea, r >> 63), c, (mc & ones) != ones);
    // Quotients at and next to the midpoint of two FP32 numbers.
    const double mid = make((rnd() & ~((1ull << 29) - 1)) | 1ull << 28, 1023 - 100 + (int)(r % 200), false);
    const double am = mid * c;
    if (std::isfinite(am) && am != 0.0) {
      check(am, c, (mc & ones) != ones);
      check(std::nextafter(am, INFINITY), c, (mc & ones) != ones);
      check(std::nextafter(am, -INFINITY), c, (mc & ones) != ones);
    }
  }
  const double special[] = {0.0, -0.0, INFINITY, -INFINITY, NAN, 5e-324, 1e308, 1e-308};
  for (double a : special)
    for (double c : {1.0, 3.0, 1e-99, 1e99, 1e-101, 1e101}) check(a, c, true);
  std::printf("%lld checked, %lld neighbours, %lld bad\n", done, neighbours, bad);
  return bad != 0;
}
"""


def test_quotients_equal_the_division(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "quotient.cpp", tmp_path / "quotient"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2606_07004_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    print(r.stdout)
