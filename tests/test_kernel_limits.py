"""The shared memory limits and resident blocks of kernels (kernel_limits.cuh)
on the host, with fake CUDA calls and two devices: the limit is raised on every
device that launches the kernel, each kernel's and each device's figures are its
own, a launch that does not fit or whose call fails is an error and is asked for
again the next time, and nothing is asked twice otherwise."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DRIVER = r"""
#include <cstdio>
#include <map>
#include "kernel_limits.cuh"

// per device: the limits set so far; 48 KB where none was
static int cur = 0, calls = 0, fail = 0;
static std::map<std::pair<int, const void*>, size_t> set_to;
struct Fake {
  using Error = int;
  static constexpr Error ok = 0, does_not_fit = 9;
  static Error device(int* d) { return *d = cur, fail == 1 ? 5 : ok; }
  static Error raise(const void* fn, size_t bytes) {
    calls++;
    if (fail == 2) return 6;
    set_to[{cur, fn}] = bytes;
    return ok;
  }
  static Error blocks(int* b, const void* fn, int threads, size_t smem) {
    calls++;
    if (fail == 3) return 7;
    const size_t sm = cur == 0 ? 228 << 10 : 100 << 10;   // the second device has less
    *b = (int)(smem ? sm / smem : 2048 / threads);
    return ok;
  }
};
// what a launch does: refused when the kernel's limit on this device is lower
static int launch(const void* fn, size_t smem) {
  const auto it = set_to.find({cur, fn});
  return smem > (it == set_to.end() ? (size_t)48 << 10 : it->second) ? 1 : 0;
}
static int bad = 0;
static void expect(bool good, const char* what) {
  if (!good && ++bad) printf("wrong: %s\n", what);
}

int main() {
  dfpr::KernelLimits<Fake> l;
  int ka, kb, b = 0;
  for (int round = 0; round < 2; round++)
    for (cur = 0; cur < 2; cur++)
      for (const void* fn : {(const void*)&ka, (const void*)&kb})
        for (size_t smem : {(size_t)0, (size_t)16 << 10, (size_t)100 << 10, (size_t)64 << 10}) {
          const int before = calls;
          expect(l.get(fn, 512, smem, &b) == 0, "status");
          expect(b == (smem ? (int)((cur == 0 ? 228u << 10 : 100u << 10) / smem) : 4), "blocks of this device");
          expect(launch(fn, smem) == 0, "the limit is raised on this device");
          expect(round == 0 || calls == before, "asked once");
        }
  cur = 1;
  expect(l.get(&ka, 512, 200 << 10, &b) == 9, "does not fit on the second device");
  cur = 0;
  expect(l.get(&ka, 512, 200 << 10, &b) == 0 && b == 1, "fits on the first");
  int fresh[4];
  for (fail = 1; fail <= 3; fail++) {
    int& k = fresh[fail];
    expect(l.get(&k, 256, 60 << 10, &b) == 4 + fail, "a failed call's status");
    const int f = fail;
    fail = 0;
    expect(l.get(&k, 256, 60 << 10, &b) == 0 && launch(&k, 60 << 10) == 0, "asked for again");
    fail = f;
  }
  printf("wrong %d\n", bad);
  return bad != 0;
}
"""


def test_limits_are_kept_per_device(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    src = tmp_path / "kernel_limits_check.cpp"
    src.write_text(DRIVER)
    exe = tmp_path / "kernel_limits_check"
    inc = os.path.join(ROOT, "paper_2401_15870_gb300", "csrc")
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-Wall", "-pthread", "-I", inc, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert "wrong 0" in r.stdout
