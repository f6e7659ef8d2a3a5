"""The exact ranking of the nearest neighbours at the edges of its register
sorts (256, 512, 1024 and 2048 survivors), with distances that binary32 cannot
tell apart, and at scales near the ends of binary32's range."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import knn_gpu, lagp        # noqa: F401

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 255, 256, 257, 512, 513, 1024, 1025, 2048, 2049]


def check(L, X, Xref, nc):
    cand = knn_gpu(L, X, Xref, nc)
    for m in range(len(Xref)):
        np.testing.assert_array_equal(cand[m], oracle.knn(X, Xref[m], nc)[0])


@pytest.mark.parametrize("nc", SIZES)
@pytest.mark.parametrize("shell", [1, 40, 64, 66, 300])
def test_knn_shells_below_binary32(lagp, nc, shell):
    """Points in shells of `shell` members around the first location, whose
    distances differ by 1e-10 relative: their order needs binary64."""
    rng = np.random.default_rng(nc + shell)
    N, p = max(2 * nc, 600), 3
    u = rng.standard_normal((N, p))
    u /= np.linalg.norm(u, axis=1)[:, None]
    k = rng.permutation(N)
    r = 0.2 + 0.5 * (k // shell) / N * shell + 1e-10 * rng.permutation(N) / N
    Xref = np.vstack([np.full(p, 0.5), rng.random((2, p))])
    check(lagp, Xref[0] + r[:, None] * u, Xref, nc)


@pytest.mark.parametrize("nc", [30, 700])
@pytest.mark.parametrize("scale", [1e-25, 1e-18, 1e-6, 1e6, 1e14])
def test_knn_scales(lagp, nc, scale):
    """At 1e-25 every binary32 distance is 0, so all 1,500 points stay in the
    running: more than the buffers of N' = 30 hold, which is reported."""
    rng = np.random.default_rng(nc)
    X, Xref = rng.random((1500, 5)) * scale, rng.random((9, 5)) * scale
    X[::3] = X[1]                                  # a run of 500 equal points
    if scale == 1e-25 and nc == 30:
        with pytest.raises(AssertionError, match="2\nassert -4 == 0"):
            check(lagp, X + 3 * scale, Xref + 3 * scale, nc)
    else:
        check(lagp, X + 3 * scale, Xref + 3 * scale, nc)
