"""The pilot thresholds of the k-nearest search, read from the workspace: the form
for small batches and the one for large ones give the same values, near the m-th
smallest sample distance; they admit what they are expected to on gridded designs
too; and the lists of large batches are the oracle's at every width of a row."""
import math

import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import to_dev
from test_gpu_parity import lagp        # noqa: F401
from test_launch_rules import values

pytestmark = pytest.mark.gpu


def search(lagp, X, xr, nc, cap):
    """Lists and thresholds of one call (the request part of a workspace starts
    with the status, the buffers, the counts and the thresholds, 256-byte
    aligned)."""
    N, p = X.shape
    M = xr.shape[0]
    ws = torch.zeros(lagp.laGP_knn_workspace_bytes(N, p, M, nc), dtype=torch.uint8, device="cuda")
    cand = torch.empty((M, nc), dtype=torch.int32, device="cuda")
    lagp.laGP_knn(X, xr, nc, cand, ws)
    assert lagp.laGP_status(ws)[0] == 0
    up = lambda x: -(-x // 256) * 256
    at = 256 + up(8 * M * cap) + up(4 * M)
    return cand.cpu().numpy(), ws[at:at + 4 * M].view(torch.float32).cpu().numpy()


def sample_rows(N):
    S = min(N // 16, 32768)
    step = N // S
    i = np.arange(S, dtype=np.uint64)
    return (i * step + (((i * 2654435769 & 0xFFFFFFFF) * step) >> np.uint64(32))).astype(np.int64)


@pytest.mark.parametrize("p", [3, 8, 11, 15])
@pytest.mark.parametrize("N,nc", [(40_053, 100), (40_053, 2000)])
def test_both_forms_and_lists(lagp, tmp_path, p, N, nc):
    """2,503 sample rows (no multiple of a tile at any width); 20,000 locations
    take the form for large batches, one alone the other. A threshold is the
    upper edge of a bin of 2^-8 of its octave, so above the m-th smallest sample
    distance by 2^-8 at most, both with the filter's binary32 error of a few 1e-6 of
    the squared distance to the farthest point."""
    cap, large, alone = values(tmp_path, ["knn_cap(%d, %d)" % (nc, N),
                                          "knn_pilot_alone(20000, %d, %d, 152)" % (N // 16, -(-p // 4) * 4),
                                          "knn_pilot_alone(1, %d, %d, 152)" % (N // 16, -(-p // 4) * 4)])
    assert (large, alone) == (0, 1)
    rng = np.random.default_rng(p + nc)
    Xh, Xr = rng.random((N, p)), rng.random((20_000, p))
    X, xr = to_dev(Xh), to_dev(Xr)
    cand, thr = search(lagp, X, xr, nc, cap)
    rows = sample_rows(N)
    lam = len(rows) * nc / N
    m = math.ceil(lam + 4.5 * math.sqrt(lam) + 4)
    for q in (0, 31, 32, 777, 19_968, 19_999):
        c1, t1 = search(lagp, X, xr[q:q + 1].contiguous(), nc, cap)
        assert t1[0] == thr[q]
        np.testing.assert_array_equal(c1[0], cand[q])
        np.testing.assert_array_equal(cand[q], oracle.knn(Xh, Xr[q], nc)[0])
        d = np.sort(((Xh[rows] - Xr[q]) ** 2).sum(1))[m - 1]
        assert d - 1e-5 * p <= thr[q] <= d * (1 + 2.0 ** -8) + 1e-5 * p


@pytest.mark.parametrize("M", [4, 3000])
@pytest.mark.parametrize("sides,nc", [((16, 16, 16), 30), ((16, 16, 16), 300), ((400, 16), 100),
                                      ((64, 64), 200)])
def test_gridded_designs(lagp, tmp_path, sides, nc, M):
    """Row-major grids whose rows are as long as the sample's step or a multiple of
    it. The design points at or below a threshold, of which the sample holds m, are
    at least N' and at most the step times m + 6 sqrt(m) + 8 (a sample of random
    rows misses that by six standard deviations)."""
    Xh = np.stack(np.meshgrid(*[np.arange(s) * 0.1 for s in sides], indexing="ij"),
                  -1).reshape(-1, len(sides))
    N = len(Xh)
    cap, = values(tmp_path, ["knn_cap(%d, %d)" % (nc, N)])
    rng = np.random.default_rng(nc)
    Xr = rng.random((M, len(sides))) * (np.array(sides) - 1) * 0.1
    cand, thr = search(lagp, to_dev(Xh), to_dev(Xr), nc, cap)
    lam = (N // 16) * nc / N
    m = math.ceil(lam + 4.5 * math.sqrt(lam) + 4)
    for q in range(0, M, max(1, M // 40)):
        np.testing.assert_array_equal(cand[q], oracle.knn(Xh, Xr[q], nc)[0])
        below = (((Xh - Xr[q]) ** 2).sum(1) <= thr[q]).sum()
        assert nc <= below <= min(16 * (m + 6 * math.sqrt(m) + 8), N), (q, below)


@pytest.mark.parametrize("M", [5, 3000])
def test_clusters_within_the_filter_s_error(lagp, tmp_path, M):
    """20 clusters of 1,000 points in a box whose filter error spans a cluster:
    a threshold would admit the cluster, more than the room of 512 entries, so
    there is none; on a uniform design there is. The lists are the oracle's."""
    rng = np.random.default_rng(M)
    N, p, nc = 20_000, 4, 30
    cap, = values(tmp_path, ["knn_cap(%d, %d)" % (nc, N)])
    Xh = rng.random((20, p))[np.arange(N) % 20] + 0.002 * rng.standard_normal((N, p))
    Xr = Xh[rng.integers(0, N, M)] + 0.001 * rng.standard_normal((M, p))
    cand, thr = search(lagp, to_dev(Xh), to_dev(Xr), nc, cap)
    assert np.isinf(thr).mean() > 0.9
    for q in range(0, M, max(1, M // 40)):
        np.testing.assert_array_equal(cand[q], oracle.knn(Xh, Xr[q], nc)[0])
    assert np.isfinite(search(lagp, to_dev(rng.random((N, p))), to_dev(Xr), nc, cap)[1]).all()
