"""Candidate searches with less room than the larger kNN buffers want: the
sizes are accepted down to the smallest buffers (CPU)."""
import ctypes as C

import pytest

N, P, M, NC = 100_000, 4, 12_000, 100       # smallest buffers 512 entries, larger ones 1,024


@pytest.fixture(scope="module")
def lib():
    from paper_1409_0074_gb300 import build
    build.build()
    from paper_1409_0074_gb300 import lagp
    L = lagp.load()
    L.laGP_knn_noalloc.restype = C.c_int
    L.laGP_knn_noalloc.argtypes = [C.c_void_p, C.c_int64, C.c_int, C.c_void_p, C.c_int64,
                                   C.c_int, C.c_void_p, C.c_void_p, C.c_void_p]
    return L


def test_noalloc_takes_what_its_scratch_holds_with_the_smallest_buffers(lib):
    """Null pointers: refused as such (-1) once the size is accepted, and before
    any device work; a size beyond the scratch is refused first (-2)."""
    scratch = 64 << 20
    want = lib.laGP_knn_workspace_bytes(N, P, M, NC)
    least = want - 8 * M * 512
    assert least <= scratch < want
    assert lib.laGP_knn_noalloc(None, N, P, None, M, NC, None, None, None) == -1
    more = M + (scratch - least) // 4096
    assert lib.laGP_knn_noalloc(None, N, P, None, more, NC, None, None, None) == -2


@pytest.mark.parametrize("n,p", [(40, 1), (64, 2), (5000, 3), (100_000, 8), (1_000_000, 16)])
def test_unlimited_scope_adds_the_tree_and_its_keys(lib, n, p):
    """The tree (order, FP32 rows, both boxes of every node) and what its sort
    takes beside it: two key buffers, one of positions, and no more than a
    kilobyte per 4,096 points."""
    from paper_1409_0074_gb300 import lagp

    def up(x):
        return (x + 255) & ~255

    size = [lib.laGP_workspace_bytes(n, p, 10, 8, 20, 2, s, lagp.LAGP_FP32_SCORE)
            for s in (lagp.LAGP_RAY, lagp.LAGP_RAY_FULL)]
    depth = 0
    while -(-n // (1 << depth)) > 32:
        depth += 1
    nodes, pp = 2 << depth, -(-p // 4) * 4
    tree = up(4 * n) + up(4 * n * pp) + up(4 * nodes * 2 * pp) + up(8 * nodes * 2 * p)
    assert size[1] - size[0] <= tree + up(16 * n) + up(4 * n) + 1024 * -(-n // 4096)
