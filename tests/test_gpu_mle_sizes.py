"""Local inference for the lengthscale at the edges of its block sizes and of its
triangular indexing: the smallest designs, odd ones, a warp and a block more or
less, the largest."""
import numpy as np
import pytest

import oracle
from gpu_helpers import to_dev
from test_gpu_parity import lagp        # noqa: F401

pytestmark = pytest.mark.gpu

G, T0, TMIN, TMAX = 1e-2, 0.3, 1e-3, 5.0


@pytest.mark.parametrize("n", [1, 2, 3, 7, 16, 23, 24, 25, 31, 32, 33, 45, 63, 64])
def test_estimate_and_prediction(lagp, n):
    """The estimate's likelihood is no lower than the oracle's estimate's, and the
    prediction is the kriging one at the estimate. Rounding of log|K| and of psi
    is at most n eps cond(K) relative (cond <= (n + g) / g), eps = 1.2e-16, with
    a factor of ten."""
    rng = np.random.default_rng(n)
    X = rng.random((400, 2))
    y = np.sin(5 * X[:, 0]) * np.cos(4 * X[:, 1]) + 0.1 * rng.standard_normal(400)
    xr = rng.random((9, 2))
    sel = np.argsort(((X[None] - xr[:, None]) ** 2).sum(-1), axis=1)[:, :n].astype(np.int32)
    import torch
    out = lagp.mle_predict(to_dev(X), to_dev(y), to_dev(xr), to_dev(sel, torch.int32), T0, G, TMIN,
                           TMAX)
    eps = 1.2e-15 * n * (n + G) / G
    for m in range(len(xr)):
        S, ys, t = X[sel[m]], y[sel[m]], float(out["theta"][m])
        assert TMIN <= t <= TMAX
        want, _ = oracle.mle_theta(S, ys, T0, G, TMIN, TMAX)
        ll, best = oracle.loglik(S, ys, t, G)[0], oracle.loglik(S, ys, want, G)[0]
        assert ll >= best - eps * (n + abs(best)), (m, t, want)
        d2 = ((S[:, None] - S[None]) ** 2).sum(-1)
        K = np.exp(-d2 / t) + G * np.eye(n)
        k = np.exp(-((S - xr[m]) ** 2).sum(1) / t)
        a, b = np.linalg.solve(K, ys), np.linalg.solve(K, k)
        assert abs(float(out["mean"][m]) - k @ a) <= eps * np.abs(k).sum() * np.abs(a).max() + 1e-14
        s2 = (ys @ a) * (1 + G - k @ b) / n
        assert abs(float(out["s2"][m]) - s2) <= eps * (ys @ a) * (1 + G) / n
