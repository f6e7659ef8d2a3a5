"""The ranking of short candidate lists, whose network is as long as the next power
of two: sizes around every one of them, with distances that binary32 cannot tell
apart and without."""
import numpy as np
import pytest

from test_gpu_parity import lagp        # noqa: F401
from test_gpu_rank_sizes import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc", [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129])
@pytest.mark.parametrize("shell", [1, 7, 66])
def test_short_lists(lagp, nc, shell):
    """Points in shells around the first location, 1e-10 apart within a shell."""
    rng = np.random.default_rng(nc + shell)
    N, p = 2 * nc + 7, 4
    u = rng.standard_normal((N, p))
    u /= np.linalg.norm(u, axis=1)[:, None]
    k = rng.permutation(N)
    r = 0.2 + 0.5 * (k // shell) / N * shell + 1e-10 * rng.permutation(N) / N
    Xref = np.vstack([np.full(p, 0.5), rng.random((3, p))])
    check(lagp, Xref[0] + r[:, None] * u, Xref, nc)
