"""Every pick of the FP32 exhaustive scorers against binary64 scores on the same
local design: it is the best candidate as far as binary32 scores can tell.

With w = L^{-1} k, z = L^{-1} k(x), a score is s = |w.z - K(c, x)| / sqrt(v), v = 1 + g -
|w|^2 (ALC = s^2). The forms' scores carry, with u = 2^-24 and all sums of magnitudes:
  k      u (4 + 2 (p + 4) d / theta + 8 sqrt(p d) / theta) |k|, from the exponential,
         the distance's arithmetic and the coordinates rounded to binary32 (within 1)
  w      |L^{-1}| dk + c (j + 4) u |L^{-1}| |k|; c = 1 (fused multiply-adds), 8 for the
         split products of the tensor-core form (3 2^-22 a product, 3 j terms)
  num    dw.|z| + (j + 4) u |w|.|z| + dK(c, x)
  v      2 |w|.dw + (j + 4) u (1 + |w|^2)
and s is off by dnum / sqrt(v) + s dv / (2 v). The pick's score plus its own and the
best one's error is at least the best one. A scorer that drops or repeats a term
of w misses that by orders of magnitude."""
import numpy as np
import pytest
from scipy.linalg import solve_triangular

from paper_1409_0074_gb300 import workloads as W
from test_gpu_exh_shapes import lagp        # noqa: F401
from test_gpu_parity import gpu_run

import oracle

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def check_picks(w, sel, m, precision):
    cand, x = oracle.knn(w.X, w.Xref[m], w.nc)[0], w.Xref[m]
    C = w.X[cand]
    rank = {int(c): r for r, c in enumerate(cand)}
    dx = ((C - x) ** 2).sum(1)
    assert list(sel[:w.n0]) == [int(c) for c in cand[:w.n0]]
    used = [rank[int(c)] for c in sel[:w.n0]]
    c = 8 if precision == "fp32_tc" and w.n <= 64 else 1

    def err_k(d):
        return U * (4 + 2 * (w.p + 4) * d / w.theta + 8 * np.sqrt(w.p * d) / w.theta)

    for j in range(w.n0, w.n):
        S = C[used]
        L = np.linalg.cholesky(np.exp(-((S[:, None] - S[None]) ** 2).sum(-1) / w.theta) +
                               w.g * np.eye(j))
        Li = np.abs(solve_triangular(L, np.eye(j), lower=True))
        d = ((S[:, None] - C[None]) ** 2).sum(-1)
        k, kx = np.exp(-d / w.theta), np.exp(-dx / w.theta)
        wc = solve_triangular(L, k, lower=True)
        z = solve_triangular(L, kx[used], lower=True)
        v, num = 1 + w.g - (wc ** 2).sum(0), z @ wc - kx
        dw = Li @ (err_k(d) * k) + c * (j + 4) * U * (Li @ k)
        dnum = np.abs(z) @ dw + (j + 4) * U * (np.abs(z) @ np.abs(wc)) + err_k(dx) * kx
        dv = 2 * (np.abs(wc) * dw).sum(0) + (j + 4) * U * (1 + (wc ** 2).sum(0))
        s = np.abs(num) / np.sqrt(v)
        e = dnum / np.sqrt(v) + s * dv / (2 * v)
        free = np.ones(w.nc, bool)
        free[used] = False
        pick = rank[int(sel[j])]
        assert free[pick], (m, j)
        best = np.flatnonzero(free)[np.argmax((s - e)[free])]
        assert s[pick] + e[pick] >= s[best] - e[best], (m, j, pick, best, s[pick], s[best])
        used.append(pick)


@pytest.mark.parametrize("precision", ["fp32", "fp32_tc"])
@pytest.mark.parametrize("n0,n,nc,M", [(3, 4, 5, 8), (3, 17, 129, 8), (16, 33, 131, 8),
                                       (17, 34, 1001, 8), (33, 64, 257, 8), (33, 64, 257, 700),
                                       (6, 65, 150, 8), (6, 50, 512, 700), (6, 40, 201, 8)])
def test_every_pick_is_a_best_one(lagp, precision, n0, n, nc, M):
    w = W.small(N=4000, p=3, M=M, n0=n0, n=n, nc=nc, theta=0.3, g=1e-2, seed=n + nc)
    g = gpu_run(lagp, w, "exhaustive", precision)
    for m in range(0, M, max(1, M // 8)):
        check_picks(w, g["selected"][m], m, precision)
