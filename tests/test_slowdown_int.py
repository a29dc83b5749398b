"""The integer form of a slowed duration (``csrc/echo_slowdown_int.h``) against llrint of the fp64 product, on the CPU:
random durations and factors, factors whose product lies on, just below and just above a half, the smallest and largest
durations and factors of its range, and what lies outside it."""
import os
import subprocess


from paper_2412_12487_gb300 import build as B

MAIN = r"""
#include "echo_slowdown_int.h"
#include <initializer_list>
#include <math.h>
#include <stdio.h>
#include <string.h>
static uint64_t state = 88172645463325252ull;
static uint64_t rnd() { state ^= state << 13; state ^= state >> 7; state ^= state << 17; return state; }
static long bad = 0, n = 0;
static void one(int64_t d, uint64_t bits) {
  double f;
  memcpy(&f, &bits, 8);
  if (!echo::slowed_int_ok(d, bits)) return;
  ++n;
  volatile double x = (double)d * f;
  if (echo::slowed_int(d, bits) != (int64_t)llrint(x) && ++bad < 10) printf("%lld %a\n", (long long)d, f);
}
int main() {
  const uint64_t one_bits = 1023ull << 52, last = one_bits | ((1ull << 52) - 1);
  for (long k = 0; k < 3000000; ++k) {
    const int64_t d = (int64_t)(rnd() >> (33 + rnd() % 31));
    one(d, one_bits | (rnd() >> 12));
    // a factor next to (i + 1/2) / d, where the product is next to a half
    if (d > 0) {
      const double t = ((double)(d + (int64_t)(rnd() % (uint64_t)d)) + 0.5) / (double)d;
      uint64_t b;
      memcpy(&b, &t, 8);
      for (int e = -3; e <= 3; ++e) one(d, b + e);
    }
    one(d, one_bits | (1ull << (rnd() % 52)));
  }
  const int64_t edge[] = {0, 1, 2, 3, (1ll << 30) - 1, 1ll << 30, (1ll << 31) - 2, (1ll << 31) - 1};
  for (int64_t d : edge)
    for (uint64_t off : {0ull, 1ull, (1ull << 52) - 2, (1ull << 52) - 1, 1ull << 51, 3ull << 50}) one(d, one_bits + off);
  const bool out = echo::slowed_int_ok(1ll << 31, one_bits) || echo::slowed_int_ok(-1, one_bits) ||
                   echo::slowed_int_ok(1, one_bits - 1) || echo::slowed_int_ok(1, last + 1) || echo::slowed_int_ok(1, last | (1ull << 63));
  printf("%ld tested, %ld wrong\n", n, bad);
  return bad || out || n < 10000000;
}
"""


def test_integer_slowdown_equals_fp64(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(B.CSRC), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
