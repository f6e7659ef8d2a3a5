"""The binary64 product on integer units (csrc/mul64.h), compiled with the host
C++ compiler and compared bit for bit with the host's own multiplication:
random significands, significands with long runs of zeros or ones (exact ties
and carries into the exponent), both signs, and the edges of the range
mul64_safe admits."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1409_0074_gb300", "csrc")

PROG = r"""
#include <cstdio>
#include <cstring>
#include <random>
#include "mul64.h"
static uint64_t bits(double d) { uint64_t u; std::memcpy(&u, &d, 8); return u; }
static double dbl(uint64_t u) { double d; std::memcpy(&d, &u, 8); return d; }
static long bad = 0, seen = 0;
static void one(uint64_t a, uint64_t b) {
  if (!lagp::mul64_safe((uint32_t)(a >> 32)) || !lagp::mul64_safe((uint32_t)(b >> 32))) return;
  ++seen;
  const uint64_t r = lagp::mul64(lagp::mul64_a((uint32_t)a, (uint32_t)(a >> 32)),
                                 lagp::mul64_b((uint32_t)b, (uint32_t)(b >> 32)));
  volatile double p = dbl(a) * dbl(b);
  if (bits(p) != r) ++bad;
}
int main() {
  std::mt19937_64 g(7);
  const uint64_t M = 0x000fffffffffffffull;
  for (long i = 0; i < 4000000; ++i) {
    uint64_t a = g() & M, b = g() & M;
    switch (i & 7) {
      case 1: a &= ~0ull << (g() % 52); b &= ~0ull << (g() % 52); break;   // trailing zeros: ties
      case 2: a |= (1ull << (g() % 52)) - 1; break;                        // trailing ones
      case 3: a |= (1ull << (g() % 52)) - 1; b |= (1ull << (g() % 52)) - 1; break;
      case 4: a |= M & ~((1ull << (g() % 52)) - 1); break;                 // leading ones
      case 5: b = 0; break;                                                // a power of two
      case 6: a = M; b = M ^ (1ull << (g() % 52)); break;                  // carries
    }
    const uint64_t ea = 524 + g() % 990, eb = 524 + g() % 990;
    one((g() & (1ull << 63)) | ea << 52 | a, eb << 52 | b);
  }
  const uint64_t lo = 0x20bull << 52, hi = (0x5f2ull << 52) | M;           // the range's ends
  one(lo, lo); one(hi, hi); one(lo, hi); one(hi | 1ull << 63, lo);
  std::printf("%ld %ld %d %d %d %d %d\n", seen, bad, lagp::mul64_safe((uint32_t)(lo >> 32)),
              lagp::mul64_safe((uint32_t)((lo - 1) >> 32)), lagp::mul64_safe((uint32_t)(hi >> 32)),
              lagp::mul64_safe((uint32_t)((hi + 1) >> 32)), lagp::mul64_safe(0));
}
"""


def test_integer_product_equals_the_binary64_product(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text(PROG)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    seen, bad, *safe = (int(v) for v in out.split())
    assert bad == 0 and seen > 3_900_000
    assert safe == [1, 0, 1, 0, 0]
