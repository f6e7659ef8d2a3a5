"""Rows that pad the design to whole tiles never become candidates, whatever the
scale of the inputs (both filters, designs that are no multiple of a tile)."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import knn_gpu, lagp        # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e14, 1e17])
@pytest.mark.parametrize("N,nc", [(300, 290), (4100, 60), (4100, 2000)])
def test_padding_rows_are_no_candidates(lagp, N, nc, scale):
    rng = np.random.default_rng(N + nc)
    X, Xref = rng.random((N, 3)) * scale, rng.random((7, 3)) * scale
    cand = knn_gpu(lagp, X, Xref, nc)
    assert cand.min() >= 0 and cand.max() < N
    for m in range(7):
        np.testing.assert_array_equal(cand[m], oracle.knn(X, Xref[m], nc)[0])
