"""The FP32 ray kernel at the edges of its row blocks and lane layouts: design
sizes around a quad, the register-held quads (32 rows) and 64 points, and ray
counts that give 2, 4, 8 and 16 lanes per ray, against the oracle."""
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


@pytest.mark.parametrize("n", [4, 5, 31, 33, 50, 66])
@pytest.mark.parametrize("nrays", [1, 3, 8, 11])
def test_fp32_ray_row_blocks(lagp, n, nrays):
    """A nugget of 1e-3 bounds cond(K) by n / g < 1e5, where FP32 scores
    resolve gaps above 1e-3 (the bar of the form's other tests)."""
    w = W.small(N=4000, p=3, M=24, n0=3, n=n, nc=150, theta=0.3, g=1e-3, seed=n + nrays,
                search="ray", nrays=nrays)
    check_fp32_form(w, gpu_run(lagp, w, "ray", "fp32"), oracle_run(w, "ray"), rmse_tol=None,
                    max_gap=1e-3)
