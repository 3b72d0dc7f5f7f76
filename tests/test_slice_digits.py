"""The 32-bit digit step of the split products' slicing, on the host.

The header is compiled with the undefined-behaviour sanitizer; for S = 3..6
slices the 64-bit digits are taken as the kernel takes them and the digits must
add up to the fixed-point value exactly, over random values and over the edges of
every digit (remainders up to the ends of the int range included)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2303_14280_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include "oz_digits.cuh"

static void check(long long v, int S) {
  const int T = 8 * S, k64 = S == 6 ? 2 : 1;
  long long r64 = v, sum = 0;
  int r = 0;
  for (int s = 0; s < S; ++s) {
    const int k = T - 8 * (s + 1);
    int d;
    if (s < k64) {
      const long long dl = (r64 + (1ll << (k - 1))) >> k;
      r64 -= dl * (1ll << k);
      d = (int)dl;
      if (s == k64 - 1) {
        if (r64 != (long long)(int)r64) std::abort();
        r = (int)r64;
      }
    } else if (k > 0) {
      d = snk::oz_take_digit(r, k);
      if (r < -(1 << (k - 1)) || r >= (1 << (k - 1))) { std::printf("remainder %d at %d\n", r, k); std::exit(1); }
    } else {
      d = r;
    }
    if (d < -256 || d > 256) { std::printf("digit %d\n", d); std::exit(1); }
    sum += (long long)d * (1ll << k);
  }
  if (sum != v) { std::printf("S %d value %lld digits give %lld\n", S, v, sum); std::exit(1); }
}

int main() {
  std::mt19937_64 g(7);
  for (int S = 3; S <= 6; ++S) {
    const long long top = 1ll << (8 * S);
    for (int n = 0; n < 2000000; ++n) check((long long)(g() % (2ull * top + 1)) - top, S);
    // remainders around the ends of the int range, after any leading digits
    for (long long lead = -3; lead <= 3; ++lead)
      for (int b = 0; b < 33; ++b)
        for (long long e = -2; e <= 2; ++e)
          for (int sg = -1; sg <= 1; sg += 2) {
            const long long v = lead * (1ll << 32) + sg * ((1ll << b) + e) + ((b & 1) ? 0x7f800000ll : 0);
            if (v >= -top && v <= top) check(v, S);
          }
    for (long long r = 0x7f7ffff0ll; r <= 0x7f800010ll; ++r)
      if (r <= top) check(r, S);
    if (S >= 5)
      for (long long r = 0x7ffffff0ll; r <= 0x80000010ll; ++r) check(r, S), check(-r, S);
  }
  return 0;
}
"""


def test_digits_add_up_without_undefined_behaviour(tmp_path):
    src, exe = tmp_path / "digits.cpp", tmp_path / "digits"
    src.write_text(SOURCE)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover=undefined",
                        "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    if r.returncode != 0 and "ubsan" in r.stderr:
        pytest.skip("no sanitizer runtime")
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
