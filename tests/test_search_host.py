"""The binary search step of the CSR check, compiled for the host: lists of
more than 2^30 entries, whose middle a 32-bit sum of both ends leaves."""
import os
import shutil
import subprocess

import pytest

from paper_2502_08042_gb300 import _native

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "kcore_search.h"
// the list 0, 1, .., len - 1: reads stay inside it and find x (or its absence) in 32 steps
static int search(int len, int x) {
  int lo = 0, hi = len;
  for (int steps = 0; steps < 33; steps++) {
    if (lo >= hi) return x >= len ? 0 : 1;
    const int mid = kc::middle(lo, hi);
    if (mid < lo || mid >= hi) return 2;
    if (mid == x) return 0;
    if (mid < x) lo = mid + 1;
    else hi = mid;
  }
  return 3;
}
int main() {
  const int lens[] = {1, 2, 3, 32, (1 << 30) - 1, 1 << 30, (1 << 30) + 1, 1500000000, 2147483645};
  for (int len : lens)
    for (int back : {-1, 0, 1, 2, 1000})
      for (int x : {back, len - 1 - back, len / 2 + back}) {
        if (x < 0) continue;
        const int r = search(len, x);
        if (r) {
          printf("len %d x %d: %d\n", len, x, r);
          return 1;
        }
      }
  return 0;
}
"""


def test_middle_of_long_lists(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "search.cpp", tmp_path / "search"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fwrapv", "-I", _native.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_the_check_uses_it():
    with open(os.path.join(_native.CSRC, "validate.cu")) as f:
        text = f.read()
    assert "middle(lo[q], hi[q])" in text and "(lo[q] + hi[q])" not in text
