"""The integer conversion of a fixed-point sum to a double (fixconv.cuh) against
the C compiler's int64 -> double conversion (IEEE 754, round to nearest even) on
the host: every power of two and its neighbours, exact halves of either parity
at every width, random values of every size, both signs and the range ends."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <cstdint>
#include <initializer_list>
#include "fixconv.cuh"

static uint64_t st = 0x9E3779B97F4A7C15ull;
static uint64_t next() {   // SplitMix64
  uint64_t z = (st += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
static long bad = 0, checked = 0;
static void one(int64_t v) {
  const double want = (double)v, got = fixconv::i64_to_f64_rn(v);
  checked++;
  if (fixconv::bits_of(want) != fixconv::bits_of(got) && bad++ < 10) printf("%lld: %a != %a\n", (long long)v, got, want);
}
static void check(uint64_t u) {
  u &= ~(1ull << 63);
  one((int64_t)u);
  one(-(int64_t)u);
}
int main() {
  check(0);
  one(INT64_MAX);
  one(INT64_MIN);
  for (int e = 0; e < 63; e++)
    for (int64_t d = -2; d <= 2; d++) check((1ull << e) + (uint64_t)d);
  for (int w = 54; w <= 63; w++)   // w-bit values: w - 53 bits are rounded off
    for (int i = 0; i < 20000; i++) {
      const uint64_t half = 1ull << (w - 54);
      const uint64_t top = (1ull << (w - 1)) | (next() >> (65 - w));
      const uint64_t kept = top & ~(2 * half - 1);
      for (uint64_t r : {half, half - 1, half + 1, (uint64_t)0, 2 * half - 1}) check(kept | r);
    }
  for (int i = 0; i < 1000000; i++) check(next() >> (next() % 64));
  printf("checked %ld, mismatches %ld\n", checked, bad);
  return bad != 0;
}
"""


def test_sum_to_double_matches_ieee_rounding(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    src = tmp_path / "to_double_check.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "to_double_check"
    inc = os.path.join(ROOT, "paper_2401_15870_gb300", "csrc")
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-I", inc, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "mismatches 0" in r.stdout
