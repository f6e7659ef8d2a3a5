"""Calls whose workspace or arena has no room for the larger kNN buffers run with
the smallest ones, with the same results; one byte less is refused."""
import ctypes as C

import numpy as np
import pytest
import torch

from gpu_helpers import to_dev
from paper_1409_0074_gb300 import workloads as W
from test_gpu_parity import lagp        # noqa: F401

pytestmark = pytest.mark.gpu

N0, N, NC, R = 4, 12, 60, 3
LESS = 8 * 512                       # bytes per location between the two buffer sizes


@pytest.fixture(scope="module")
def w():
    return W.small(N=20_000, p=3, M=333, n0=N0, n=N, nc=NC, theta=0.3, g=1e-4, seed=5, nrays=R)


def test_entry_points_that_take_a_workspace(lagp, w):
    X, Y, xr = to_dev(w.X), to_dev(w.Y), to_dev(w.Xref)
    M, pr = w.M, lagp.LAGP_FP32_SCORE
    shape = (w.N, w.p, M, N, NC, R, lagp.LAGP_RAY, pr)
    full = lagp.laGP_workspace_bytes(*shape)
    outs = []
    for wsb in (full, full - LESS * M):
        mean, s2 = torch.zeros(M, dtype=torch.float64, device="cuda"), torch.zeros(
            M, dtype=torch.float64, device="cuda")
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        go = (X, Y, xr, N0, N, NC, w.theta, w.g, lagp.LAGP_RAY, R, pr, mean, s2)
        lagp.laGP_build_and_predict(*go, ws)
        assert lagp.laGP_status(ws)[0] == 0
        outs.append((mean.clone(), s2.clone()))
        plan = lagp.Plan(*go, ws)
        mean.zero_()
        plan.launch()
        assert lagp.laGP_status(ws)[0] == 0
        plan.close()
        assert torch.equal(mean, outs[0][0]) and torch.equal(s2, outs[0][1])
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    with pytest.raises(lagp.LagpError) as e:
        lagp.laGP_build_and_predict(*go, ws[:-1])
    assert e.value.rc == -2
    # candidates alone, and the fixed scratch
    lists = []
    for less in (0, LESS * M):
        ws = torch.empty(lagp.laGP_knn_workspace_bytes(w.N, w.p, M, NC) - less, dtype=torch.uint8,
                         device="cuda")
        cand = torch.full((M, NC), -7, dtype=torch.int32, device="cuda")
        lagp.laGP_knn(X, xr, NC, cand, ws)
        assert lagp.laGP_status(ws)[0] == 0
        lists.append(cand)
    assert torch.equal(*lists)
    # local inference, and host buffers
    for less in (0, LESS * M):
        ws = torch.empty(lagp.laGP_mle_workspace_bytes(*shape) - less, dtype=torch.uint8,
                         device="cuda")
        th, mean, s2 = (torch.zeros(M, dtype=torch.float64, device="cuda") for _ in range(3))
        lagp.laGP_build_and_predict_mle(X, Y, xr, N0, N, NC, w.theta, w.g, 1e-3, 10.0, 2,
                                        lagp.LAGP_RAY, R, pr, th, mean, s2, ws)
        assert lagp.laGP_status(ws)[0] == 0
        if less == 0:
            want = th.clone(), mean.clone(), s2.clone()
    assert all(torch.equal(a, b) for a, b in zip(want, (th, mean, s2)))
    full = lagp.laGP_host_workspace_bytes(*shape)
    hm, hs = np.zeros(M), np.zeros(M)
    f = lagp.load().laGP_build_and_predict_host
    a = [np.ascontiguousarray(v) for v in (w.X, w.Y, w.Xref)]
    for less, rc in ((LESS * M, 0), (LESS * M + 256, -2)):
        ws = torch.empty(full - less, dtype=torch.uint8, device="cuda")
        assert f(a[0].ctypes.data, a[1].ctypes.data, w.N, w.p, a[2].ctypes.data, M, N0, N, NC,
                 w.theta, w.g, lagp.LAGP_RAY, R, pr, None, None, hm.ctypes.data, hs.ctypes.data,
                 None, None, None, ws.data_ptr(), ws.numel(), None) == rc
    np.testing.assert_array_equal(hm, outs[0][0].cpu().numpy())


def test_fixed_scratch_beyond_the_larger_buffers(lagp):
    """12,000 locations whose larger buffers exceed the library's 64 MiB array:
    the lists of laGP_knn."""
    rng = np.random.default_rng(2)
    n, p, m, nc = 100_000, 4, 12_000, 100
    X, xr = to_dev(rng.random((n, p))), to_dev(rng.random((m, p)))
    ws = torch.empty(lagp.laGP_knn_workspace_bytes(n, p, m, nc), dtype=torch.uint8, device="cuda")
    want = torch.empty((m, nc), dtype=torch.int32, device="cuda")
    lagp.laGP_knn(X, xr, nc, want, ws)
    assert lagp.laGP_status(ws)[0] == 0
    f = lagp.load().laGP_knn_noalloc
    f.restype = C.c_int
    f.argtypes = [C.c_void_p, C.c_int64, C.c_int, C.c_void_p, C.c_int64, C.c_int, C.c_void_p,
                  C.c_void_p, C.c_void_p]
    cand = torch.full((m, nc), -7, dtype=torch.int32, device="cuda")
    st = torch.full((1,), 77, dtype=torch.int32, device="cuda")
    assert f(X.data_ptr(), n, p, xr.data_ptr(), m, nc, cand.data_ptr(), st.data_ptr(),
             torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert int(st.item()) == 0 and torch.equal(cand, want)


def test_context_whose_arena_holds_the_smaller_request_only(lagp, w):
    X, Y = to_dev(w.X), to_dev(w.Y)
    L, pr = lagp.load(), lagp.LAGP_FP32_SCORE
    d = L.laGP_ctx_design_bytes(w.N, w.p)
    rb = L.laGP_ctx_request_bytes(w.N, w.p, w.M, N, NC, R, lagp.LAGP_RAY, pr, 0)
    out = []
    for room in (rb, rb - LESS * w.M, rb - LESS * w.M - 256):
        ctx = lagp.Context(X, Y, w.theta, w.g, N0, NC, lagp.LAGP_RAY, R, pr, d + room,
                           max_inflight=2)
        mean = torch.zeros(w.M, dtype=torch.float64).pin_memory().numpy()
        s2 = torch.zeros(w.M, dtype=torch.float64).pin_memory().numpy()
        t = ctx.submit(np.ascontiguousarray(w.Xref), N, mean, s2)
        if room < rb - LESS * w.M:
            assert t is None
        else:
            ctx.wait(t)
            out.append((mean.copy(), s2.copy()))
        ctx.close()
    np.testing.assert_array_equal(out[0], out[1])
