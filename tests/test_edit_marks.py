"""The marks the row edit keeps per old element of a chunk (edit_marks.cuh), on
the host: where every surviving element goes, against a merge of the lists, for
random chunks with many and few changes, and with numbers of insertions in front
of one element around every power of two up to what a row can hold (ids are
below 2^31): the element stays, and it and those behind it move by that many."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <cstdint>
#include <set>
#include <vector>
#include "edit_marks.cuh"
using namespace editmarks;

static uint64_t st = 0x9E3779B97F4A7C15ull;
static uint64_t next() {   // SplitMix64
  uint64_t z = (st += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
static long bad = 0, checked = 0;
static void expect(bool ok, const char* what, long a, long b) {
  checked++;
  if (!ok && bad++ < 10) printf("%s: %ld %ld\n", what, a, b);
}

int main() {
  const int LEN = 1024;
  std::vector<int32_t> shift(LEN + 1);
  std::vector<uint32_t> dead(LEN / 32);
  auto clear = [&] { shift.assign(LEN + 1, 0), dead.assign(LEN / 32, 0u); };
  // old elements 10, 20, ..: an insertion in front of element i is any value
  // between its neighbours
  for (int trial = 0; trial < 200; trial++) {
    clear();
    const int no = 1 + (int)(next() % LEN);
    std::vector<int> ins(no + 1), del(no);
    for (int i = 0; i < no; i++) del[i] = next() % 4 == 0;
    for (int k = (int)(next() % 5000); k > 0; k--) ins[trial % 2 ? next() % (no + 1) : (uint64_t)no / 2]++;
    for (int i = 0; i <= no; i++)
      for (int k = 0; k < ins[i]; k++) mark_inserted(shift.data(), i, 1);
    for (int i = 0; i < no; i++)
      if (del[i]) mark_deleted(shift.data(), dead.data(), i);
    long at = 0, sum = 0;   // merged position, running shift
    for (int i = 0; i < no; i++) {
      at += ins[i];
      sum += shift[i];
      expect(is_deleted(dead.data(), i) == (bool)del[i], "deleted", i, del[i]);
      if (!del[i]) expect(i + sum == at++, "position", i + sum, at);
    }
  }
  // crowds: k insertions in front of element 7, elements 3 and 7 deleted or not
  for (int e = 0; e <= 31; e++)
    for (int64_t d = -2; d <= 2; d++) {
      const int64_t k = (1ll << e) + d;
      if (k < 0 || k > INT32_MAX - 16) continue;
      for (int mask = 0; mask < 4; mask++) {
        clear();
        mark_inserted(shift.data(), 7, (int32_t)(k / 2));
        if (mask & 1) mark_deleted(shift.data(), dead.data(), 3);
        if (mask & 2) mark_deleted(shift.data(), dead.data(), 7);
        mark_inserted(shift.data(), 7, (int32_t)(k - k / 2));
        int64_t sum = 0;
        for (int i = 0; i < 16; i++) {
          sum += shift[i];
          const bool gone = (i == 3 && (mask & 1)) || (i == 7 && (mask & 2));
          expect(is_deleted(dead.data(), i) == gone, "crowd deleted", (long)k, i);
          const int64_t want = i + (i >= 7 ? k : 0) - ((mask & 1) && i > 3) - ((mask & 2) && i > 7);
          expect(i + sum == want, "crowd position", (long)(i + sum), (long)want);
        }
      }
    }
  printf("checked %ld, mismatches %ld\n", checked, bad);
  return bad != 0;
}
"""


def test_marks_of_a_chunk_match_a_merge(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    src = tmp_path / "edit_marks_check.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "edit_marks_check"
    inc = os.path.join(ROOT, "paper_2401_15870_gb300", "csrc")
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-Wall", "-I", inc, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "mismatches 0" in r.stdout
