"""Which form of a kernel a call takes (csrc/launch_plan.h), compiled with the host
C++ compiler and checked on the CPU against the sides that were measured."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1409_0074_gb300", "csrc")


def values(tmp_path, expressions):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    body = "".join('  std::printf("%%lld\\n", (long long)(%s));\n' % e for e in expressions)
    src.write_text('#include <cstdio>\n#include "launch_plan.h"\nusing namespace lagp;\n'
                   "int main() {\n%s}\n" % body)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    return [int(v) for v in out.split()]


def test_local_inference_of_small_designs_takes_small_blocks(tmp_path):
    """With 256 threads, 10,000 designs of 2 to 10 points took 1.4 to 1.75 times
    as long as with 128."""
    got = values(tmp_path, ["mle_threads(%d)" % n for n in (1, 2, 10, 24, 28, 50, 64)])
    assert got == [128, 128, 128, 128, 256, 256, 256]


def test_short_lists_are_ranked_by_small_blocks(tmp_path):
    """With 256 threads and a network of 256, lists of 30 took twice as long."""
    got = values(tmp_path, ["rank_threads(%d)" % n for n in (1, 30, 100, 128, 200, 1000, 4096)])
    assert got == [128, 128, 128, 128, 256, 256, 256]


def test_pilot_takes_a_block_per_location_where_that_was_faster(tmp_path):
    """(M, S, PP): a block per location lost at small samples (one location at
    S = 68 23 against 12 us) and at many locations, and won at large samples."""
    sides = {(1, 68, 4): 0, (32, 312, 4): 0, (300, 1875, 4): 0, (1000, 6250, 4): 0, (304, 1250, 8): 0,
             (608, 6250, 8): 0, (10_000, 32768, 8): 0, (1, 1875, 4): 1, (300, 6250, 4): 1,
             (152, 1250, 8): 1, (456, 6250, 8): 1, (1, 32768, 8): 1, (1024, 32768, 8): 1}
    got = values(tmp_path, ["knn_pilot_alone(%d, %d, %d, 152)" % k for k in sides])
    assert got == list(sides.values())


def test_exhaustive_scorer_takes_small_blocks_for_few_candidates(tmp_path):
    """(M, N'): four blocks of 256 threads per SM ran 700 locations at N' = 100 in
    two waves, 1.33 times as long as six had in one."""
    sides = {(700, 100): 128, (1, 60): 128, (20_000, 200): 128, (20_000, 512): 128, (700, 300): 128,
             (300, 256): 256, (1, 512): 256, (20_000, 1000): 256, (700, 1000): 256}
    got = values(tmp_path, ["d32_threads(%d, %d, 152)" % k for k in sides])
    assert got == list(sides.values())


def test_small_binary64_batches_use_the_pipe_s_products(tmp_path):
    """(M, N'): one warp with candidates per sub-partition waits for the products,
    which the integer units form later (1.25 and 1.38 ms of kernel at N' = 60)."""
    sides = {(1, 60): 0, (152, 128): 0, (304, 60): 0, (100, 200): 1, (153, 100): 1, (456, 60): 1,
             (2000, 30): 1, (1, 1000): 1}
    got = values(tmp_path, ["d64_ints(%d, %d, 152)" % k for k in sides])
    assert got == list(sides.values())


def test_few_candidates_in_binary64_take_small_blocks(tmp_path):
    """(M, n, N'): with eight warps whatever N', 1,300 locations at n = N' = 30 took
    1.31 times as long as before their blocks needed more registers."""
    sides = {(1300, 30, 30): 4, (1, 30, 60): 4, (2000, 100, 128): 4, (900, 50, 60): 4,
             (400, 50, 60): 8, (1, 60, 90): 8, (2000, 50, 1000): 8, (2000, 20, 129): 8}
    got = values(tmp_path, ["d64_warps(%d, %d, %d, 152)" % k for k in sides])
    assert got == list(sides.values())
