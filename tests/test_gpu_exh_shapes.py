"""The FP32 exhaustive scorers at the edges of their layouts, against the
oracle: design sizes around four rows, the shared-memory factor's limit (64
points) and the tensor-core form's blocks of 16 rows (also with more starting
points than one block), and candidate counts that are no multiple of four or
of a 128-candidate tile."""
import pytest

from gpu_helpers import check_fp32_form
from paper_1409_0074_gb300 import workloads as W
from test_gpu_parity import gpu_run, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lagp(cuda):
    from paper_1409_0074_gb300 import build
    build.build()
    from paper_1409_0074_gb300 import lagp as L
    L.load()
    return L


@pytest.mark.parametrize("precision", ["fp32", "fp32_tc"])
@pytest.mark.parametrize("n0,n,nc", [(3, 4, 5), (3, 17, 129), (16, 33, 131), (17, 34, 1001),
                                     (33, 64, 257), (6, 65, 1150)])
def test_fp32_exhaustive_shapes(lagp, precision, n0, n, nc):
    """With a nugget of 1e-2 the pivots are at least 1e-2, so the FP32 error of
    a few 1e-7 in a score's denominator moves scores by less than 1e-4: designs
    may leave the oracle's only at gaps below 1e-3."""
    w = W.small(N=4000, p=3, M=20, n0=n0, n=n, nc=nc, theta=0.3, g=1e-2, seed=n + nc)
    check_fp32_form(w, gpu_run(lagp, w, "exhaustive", precision), oracle_run(w, "exhaustive"),
                    rmse_tol=None, max_gap=1e-3)
