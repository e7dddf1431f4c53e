"""The integer-pipe FP64 division and square root (csrc/int64div.cuh) against
IEEE arithmetic on the host: random and hard significands (all ones, equal,
one unit apart, perfect squares and their neighbours), exponents over the
whole range (zeros, subnormals, overflow), and seeds off by up to 2^-22."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "int64div.cuh"
#include <cmath>
#include <cstdio>
#include <cstdlib>
namespace mhd { namespace i64 {
static double off = 0.0;
static float rcp(float f) { return (float)(1.0 / f * (1.0 + off)); }
static float rsq(float f) { return (float)(1.0 / std::sqrt((double)f) * (1.0 + off)); }
float (*seed_rcp)(float) = rcp;
float (*seed_rsqrt)(float) = rsq;
} }
using namespace mhd::i64;
static uint64_t st;
static uint64_t rnd() {  // splitmix64
  uint64_t z = (st += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
static bool same(double x, double y) { return bits(x) == bits(y) || (std::isnan(x) && std::isnan(y)); }
int main(int argc, char** argv) {
  const int mode = std::atoi(argv[1]);
  st = 1000 + mode;
  const uint64_t M = 0xfffffffffffffull;
  long bad = 0;
  for (int i = 0; i < 1500000; ++i) {
    if (i % 500 == 0) off = (i % 1500 == 0 ? (i & 1 ? 1.0 : -1.0) : (rnd() >> 11) * 0x1p-52 - 1.0) * 0x1p-22;
    uint64_t a = rnd(), b = rnd();
    uint64_t ma = a & M, mb = b & M, ea = 700 + (a >> 54) % 600, eb = 700 + (b >> 54) % 600;
    if (mode == 1) mb = i & 1 ? M : 0;
    if (mode == 2) ma = (mb + i % 7 - 3) & M;
    if (mode == 3) { ma = M - i % 5; mb &= ~0xffffffffull; }
    if (mode == 4) { ma >>= 20; mb |= 0xffffffull; }
    if (mode == 5) { ea = (a >> 52) & 0x7ff; eb = (b >> 52) & 0x7ff; }
    double x = value((a & 1ull << 63) | ea << 52 | ma), y = value((b & 1ull << 63) | eb << 52 | mb);
    if (mode == 5 && i % 5 == 0) x *= 0.0;
    if (mode == 5 && i % 9 == 0) y *= 0.0;
    double r = std::fabs(x);
    if (mode == 6) {  // squares and their neighbours
      r = std::sqrt(r);
      r = value(bits(r) & ~0x7ffffffull);
      r = r * r;
      if (i % 3) r = std::nextafter(r, i % 3 == 1 ? 1e300 : 0.0);
    }
    bad += !same(div(x, y), x / y) + !same(div_scaled<1>(x, y), (x + x) / y) + !same(div(1.0, y), 1.0 / y);
    bad += !same(sqrt_rn(r), std::sqrt(r)) + !same(sqrt_rn(x), std::sqrt(x));
    bad += !same(scale<-1>(x), 0.5 * x) + !same(scale<-2>(x), 0.25 * x) + !same(scale<1>(x), 2 * x) + !same(scale<2>(x), 4 * x);
    bad += (pos(x) != (x > 0)) + (neg(x) != (x < 0)) + (ge0(x) != (x >= 0)) + (abs_gt(x, std::fabs(y)) != (std::fabs(x) > std::fabs(y)) && !std::isnan(y));
    if (std::isfinite(x) && std::isfinite(y)) {
      const double t = std::fabs(x * 0.5), m = std::fmax(std::fabs(y), t);
      bad += clearly_above(x, t, 1.0, std::fabs(y)) && !(std::fabs(x) > 1e-12 * m);
      bad += clearly_above(x, y, y, t) && y * y < 1e300 && !(std::fabs(x) > 1e-12 * std::fmax(y * y, t));
    }
  }
  std::printf("%ld\n", bad);
  return bad != 0;
}
"""


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    d = tmp_path_factory.mktemp("int64div")
    (d / "t.cpp").write_text(SRC)
    exe = str(d / "t")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1112_1710_gb300", "csrc"), str(d / "t.cpp"),
                    "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("mode", range(7))
def test_int64_division_and_root_are_ieee(prog, mode):
    r = subprocess.run([prog, str(mode)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout
