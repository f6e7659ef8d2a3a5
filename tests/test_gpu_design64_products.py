"""Binary64 exhaustive designs with products from the binary64 pipe (a few small
locations) and from the integer units: the same bits, and the oracle's."""
import numpy as np
import pytest

from paper_1409_0074_gb300 import workloads as W
from test_gpu_parity import assert_fp64_parity, gpu_run, lagp, oracle_run        # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc", [25, 60, 64, 65, 128, 129])
def test_batches_on_both_sides_of_the_rule_agree(lagp, nc):
    w = W.small(N=1500, p=3, M=500, n0=4, n=20, nc=nc, theta=0.1, g=1e-4, seed=nc)
    big = gpu_run(lagp, w, "exhaustive", "fp64")           # four locations per SM
    for M in (300, 6):
        w.Xref, w.M = w.Xref[:M], M
        g = gpu_run(lagp, w, "exhaustive", "fp64")
        for k in ("selected", "mean", "s2", "tie_gap"):
            np.testing.assert_array_equal(g[k], big[k][:M])
    ident, _ = assert_fp64_parity(g, oracle_run(w, "exhaustive"), w.n0, w.M)
    assert ident == w.M
