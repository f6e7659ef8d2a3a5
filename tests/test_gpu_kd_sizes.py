"""The k-d tree's sort at the edges of its tiles of 1,024 keys."""
import numpy as np
import pytest

from paper_1409_0074_gb300 import workloads as W
from test_gpu_parity import assert_fp64_parity
from test_gpu_ray_full import lagp, oracle_full, run_full        # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1023, 1024, 1025, 2049])
@pytest.mark.parametrize("flat", [False, True])
def test_full_scope_sort_tiles(lagp, N, flat):
    """Designs with the unlimited scope equal to the oracle's; `flat`: one
    coordinate the same everywhere (a box without extent) and another on 5 values."""
    w = W.small(N=N, p=3, M=6, n0=3, n=12, nc=40, theta=0.1, g=1e-4, seed=N, nrays=3)
    if flat:
        w.X[:, 0] = w.Xref[:, 0] = 0.25
        w.X[:, 1] = np.round(w.X[:, 1] * 4) / 4
    g = run_full(lagp, w, "fp64", 3)
    ident, _ = assert_fp64_parity(g, oracle_full(w, 3), w.n0, w.M)
    assert ident >= w.M - 1
