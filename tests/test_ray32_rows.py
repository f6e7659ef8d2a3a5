"""Storage of the FP32 inverse factor in the ray kernel (csrc/ray32_layout.h),
compiled with the host C++ compiler: for every design size, each element of
the rows (padded to quads) has its own word inside the region, a row's quads
are a constant stride apart, and blocks of four rows keep their rows' quads
side by side (the unrolled product reads rows below 32 at the full stride)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1409_0074_gb300", "csrc")

PROG = r"""
#include <cstdio>
#include <set>
#define KD_STACK 64
#include "ray32_layout.h"
using namespace lagp;
int main() {
  for (int n = 1; n <= 128; ++n) {
    std::set<int> seen;
    int bad = 0;
    for (int i = 0; i < n; ++i) {
      const int u = i >> 2, st = lf_stride(u, n);
      if (u < 8 && st != 16) bad |= 1;
      for (int k = 0; k <= (i | 3); ++k) {
        const int a = lf_at(i, k, n);
        if (a < 0 || a >= lf_words(n)) bad |= 2;
        if (!seen.insert(a).second) bad |= 4;
        if (a != lf_block(u) + 4 * (i & 3) + st * (k >> 2) + (k & 3)) bad |= 8;
      }
    }
    std::printf("%d %d %d %d\n", n, bad, lf_words(n), roff(n));
  }
}
"""


def test_every_element_has_its_own_word(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "r.cpp", tmp_path / "r"
    src.write_text(PROG)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    rows = [tuple(int(v) for v in l.split()) for l in
            subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert [r[0] for r in rows] == list(range(1, 129))
    for n, bad, words, padded in rows:
        assert bad == 0, (n, bad)
        # past 32 rows the region is as large as rows padded to quads
        assert words == padded if n > 32 or n % 4 == 0 else words >= padded
