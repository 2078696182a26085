"""Index arithmetic of the kernels, compiled for the host. The binary search
step of the CSR check: lists of more than 2^30 entries, whose middle a 32-bit
sum of both ends leaves. The batched peel's chunks: 1,024 lists of more than
2^21 arcs, whose 32-bit sum overflows."""
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
static int chunks() {
  for (int block : {256, 512, 1024})
    for (long long dmax : {0ll, 1ll, 65535ll, 2097151ll, 2097152ll, 4194305ll, 1ll << 30, 2147483645ll}) {
      const long long c = kc::chunk_vertices(block, (int)dmax);
      if (c < 1 || c > block || c * dmax > 0x7fffffff || (c < block && (c + 1) * dmax <= 0x7fffffff)) {
        printf("block %d dmax %lld: %lld\n", block, dmax, c);
        return 1;
      }
    }
  return 0;
}
int main() {
  if (chunks()) return 1;
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


def test_middle_and_chunks(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "search.cpp", tmp_path / "search"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fwrapv", "-I", _native.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_the_kernels_use_them():
    with open(os.path.join(_native.CSRC, "validate.cu")) as f:
        text = f.read()
    assert "middle(lo[q], hi[q])" in text and "(lo[q] + hi[q])" not in text
    with open(os.path.join(_native.CSRC, "batched.cu")) as f:
        text = f.read()
    assert text.count("= chunk_vertices(BLOCK, dmax);") == 2 and text.count("min(chunk, nf - c0)") == 2
