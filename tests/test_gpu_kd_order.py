"""The k-d tree separates the points of every node by its split coordinate, as far as
the FP32 rows do: also where a design has half its points within 1e-8 of the centre of
its box, and where all are within a narrow band beside two far ones."""
import numpy as np
import pytest
import torch

from gpu_helpers import to_dev
from test_gpu_parity import lagp        # noqa: F401

pytestmark = pytest.mark.gpu


def order(lagp, X):
    """Tree position -> design index, the first piece of the tree, which ends the
    workspace of a call with the unlimited scope."""
    N, p = X.shape
    up = lambda x: -(-x // 256) * 256
    depth = 0
    while -(-N // (1 << depth)) > 32:
        depth += 1
    nodes, pp = 2 << depth, -(-p // 4) * 4
    tree = (up(4 * N) + up(4 * N * pp) + up(8 * nodes * pp) + up(16 * nodes * p) + up(16 * N) +
            up(4 * N) + 1024)
    shape = (N, p, 2, 3, 20, 1, lagp.LAGP_RAY_FULL, lagp.LAGP_FP32_SCORE)
    ws = torch.empty(lagp.laGP_workspace_bytes(*shape), dtype=torch.uint8, device="cuda")
    d, y, xr = to_dev(X), to_dev(X[:, 0].copy()), to_dev(X[:2] + 0.5)
    mean, s2 = (torch.empty(2, dtype=torch.float64, device="cuda") for _ in range(2))
    lagp.laGP_build_and_predict(d, y, xr, 2, 3, 20, 0.5, 1e-2, lagp.LAGP_RAY_FULL, 1,
                                lagp.LAGP_FP32_SCORE, mean, s2, ws)
    torch.cuda.synchronize()
    at = ws.numel() - tree
    return ws[at:at + 4 * N].view(torch.int32).cpu().numpy(), depth


@pytest.mark.parametrize("kind", ["uniform", "core", "band"])
@pytest.mark.parametrize("N,p", [(3000, 2), (5001, 3)])
def test_every_split_separates(lagp, kind, N, p):
    rng = np.random.default_rng(N)
    X = rng.uniform(-1, 1, (N, p))
    if kind == "core":
        X[: N // 2] = 1e-8 * rng.standard_normal((N // 2, p))
    if kind == "band":
        X *= 1e-9
    X[-1], X[-2] = 1.0, -1.0
    perm, depth = order(lagp, X)
    np.testing.assert_array_equal(np.sort(perm), np.arange(N))
    rows = (X - 0.5 * (X.min(0) + X.max(0))).astype(np.float32)[perm]
    nodes = [(0, N)]
    for level in range(depth):
        c, nxt = rows[:, level % p], []
        for a, b in nodes:
            m = (a + b) // 2
            assert c[a:m].max() <= c[m:b].min(), (level, a, b)
            nxt += [(a, m), (m, b)]
        nodes = nxt
