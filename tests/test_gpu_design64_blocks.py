"""Binary64 exhaustive designs from blocks of 512 threads (small batches) and of
256: the same bits, and the oracle's, at the edges of the threads' candidates."""
import numpy as np
import pytest

from paper_1409_0074_gb300 import workloads as W
from test_gpu_parity import assert_fp64_parity, gpu_run, lagp, oracle_run        # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc", [256, 257, 512, 513, 1030])
def test_small_and_large_batches_agree(lagp, nc):
    w = W.small(N=1500, p=2, M=180, n0=4, n=20, nc=nc, theta=0.1, g=1e-4, seed=nc)
    big = gpu_run(lagp, w, "exhaustive", "fp64")           # more locations than SMs
    w.Xref, w.M = w.Xref[:6], 6
    g = gpu_run(lagp, w, "exhaustive", "fp64")
    for k in ("selected", "mean", "s2", "tie_gap"):
        np.testing.assert_array_equal(g[k], big[k][:6])
    ident, _ = assert_fp64_parity(g, oracle_run(w, "exhaustive"), w.n0, w.M)
    assert ident == w.M
