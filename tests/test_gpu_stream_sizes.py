"""The k-nearest streams around the sizes where their form changes: a pilot
threshold from N >= max(4 N', 1024) on where the buffers have room for what it
passes, and the tensor cores from N >= 32 N'."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import knn_gpu, lagp        # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["uniform", "grid", "sampled_rows_near"])
@pytest.mark.parametrize("p,N,M,nc", [(3, 1023, 20, 200), (3, 1024, 1, 256), (8, 2799, 40, 700),
                                      (8, 2800, 40, 700), (2, 9599, 33, 300), (2, 9600, 33, 300)])
def test_knn_around_the_pilot_rule(lagp, p, N, M, nc, kind):
    """Lists equal to the oracle's: on uniform points, on a coarse grid (many
    equal distances, which go to the lower index) and where the pilot's sample
    is a cluster at the locations (its threshold is too tight: streamed again).
    The 2-d grid has 49 places, with up to 1,394 points within the 300th
    distance, which a location's buffer has to hold."""
    rng = np.random.default_rng(N + nc)
    X, Xref = rng.random((N, p)), rng.random((M, p))
    if kind == "grid":
        X, Xref = np.round(X * 6) / 8, np.round(Xref * 6) / 8
    if kind == "sampled_rows_near":
        S = N // 16
        X[np.arange(S) * (N // S)] = 0.5 + 0.01 * rng.standard_normal((S, p))
        Xref = 0.5 + 0.01 * rng.standard_normal((M, p))
    cand = knn_gpu(lagp, X, Xref, nc)
    for m in range(M):
        idx, _ = oracle.knn(X, Xref[m], nc)
        np.testing.assert_array_equal(cand[m], idx)
