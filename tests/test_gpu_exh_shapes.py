"""The FP32 exhaustive scorers at the edges of their layouts: design sizes
around four rows, the shared-memory factor's limit (64 points) and the
tensor-core form's blocks of 16 rows (also with more starting points than one
block), and candidate counts that are no multiple of four or of a 128-candidate
tile."""
import numpy as np
import pytest

from gpu_helpers import check_fp32_form, to_dev
from paper_1409_0074_gb300 import workloads as W
from test_gpu_parity import gpu_run, oracle_run, same_rows

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
    """The binary64 update and prediction on the form's own designs, s2 where
    the designs are the oracle's, and the same bits from a call whose largest
    n and N' are above every location's (other strides and tiles, and for n
    <= 64 the factor in global instead of shared memory)."""
    w = W.small(N=4000, p=3, M=20, n0=n0, n=n, nc=nc, theta=0.3, g=1e-2, seed=n + nc)
    g = gpu_run(lagp, w, "exhaustive", precision)
    check_fp32_form(w, g, oracle_run(w, "exhaustive"), rmse_tol=None, max_gap=None)
    import torch
    big = lagp.predict(to_dev(w.X), to_dev(w.Y), to_dev(w.Xref), n0, min(n + 67, 128), nc + 141, w.theta,
                       w.g, search="exhaustive", precision=precision, want_trace=True,
                       n_loc=to_dev(np.full(w.M, n, np.int32), torch.int32),
                       nclose_loc=to_dev(np.full(w.M, nc, np.int32), torch.int32))
    b = {k: v.cpu().numpy() for k, v in big.items()}
    b["selected"] = b["selected"][:, :n]
    if precision == "fp32_tc" and n > 64:
        return                  # both calls take the CUDA-core scorer: covered by "fp32"
    assert same_rows(g, b).all()
