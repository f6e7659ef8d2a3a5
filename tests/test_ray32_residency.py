"""What the k-d walk's scratch and the row storage take of a warp's shared memory
in the ray kernel (csrc/ray32_layout.h), on the CPU: the scratch costs no warp of
an SM at any shape (the limited scope has it too and runs no walk), and the rows
of the inverse factor, as the product reads them, stay inside their region."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1409_0074_gb300", "csrc")

PROG = r"""
#include <cstdio>
#include <initializer_list>
#include "launch_plan.h"
#include "ray32_layout.h"
using namespace lagp;
static int resident(size_t wb) {
  int best = 0;
  for (int rw = 1; rw <= 4; rw *= 2) {
    int ctas = (int)(233472 / (rw * wb + 1024));
    if (ctas > 20 / rw) ctas = 20 / rw;
    if (ctas * rw > best) best = ctas * rw;
  }
  return best;
}
int main() {
  for (int n = 1; n <= 128; ++n)
    for (int RP : {2, 4, 8, 16})
      for (int PP : {4, 8, 12, 16})
        for (int nc = n; nc <= 4096; nc += nc < 512 ? 37 : 256) {
          const WarpLayout w = warp_layout(n, PP, RP, nc);
          const int cbw = 2 * RP * kz_ld(n), cb = w.zf - w.cb;
          std::printf("%d %d %d %d %d %d %d %d %d\n", n, RP, PP, nc, resident(w.bytes),
                      resident(w.bytes - 4 * (cb - cbw)), cb - 33 * KD_STACK, w.kz - w.lf,
                      lf_words(n));
        }
}
"""


def test_residency_and_rows(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    kd = re.search(r"#define KD_STACK (\d+)", open(os.path.join(CSRC, "kdtree.cuh")).read())
    src, exe = tmp_path / "r.cpp", tmp_path / "r"
    src.write_text(PROG)
    subprocess.run([cxx, "-std=c++17", "-O1", "-DKD_STACK=" + kd.group(1), "-I", CSRC, str(src),
                    "-o", str(exe)], check=True)
    rows = [tuple(map(int, l.split())) for l in
            subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) > 10_000
    for n, rp, pp, nc, have, without, walk, lf, words in rows:
        assert have == without, (n, rp, pp, nc, have, without)
        assert walk >= 0 and lf >= words, (n, rp, pp, nc)
