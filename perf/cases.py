"""Cases for timing the framework through its public entry points.

Each case is one call a user's program makes: a batch prediction on device
buffers, a request to the serving context, a replayed plan, the candidate
search alone, local designs coupled with local inference for the lengthscale,
and the global fit that pre-scales the inputs.  Sizes follow the repository's
workloads (workloads.py, bench.py) and its tests.

`exact` restates the method in plain torch binary64 (incremental Cholesky
factor, batched Brent searches), independent of the package.
"""
import math

import numpy as np
import torch

from paper_1409_0074_gb300 import lagp

DEV = "cuda"


def _case(name, kind, N, p, M, n, nc, search="ray", nrays=0, precision="fp32", n0=6, theta=None,
          g=1e-6, response="sinusoid", stages=2):
    return dict(name=name, kind=kind, N=N, p=p, M=M, n0=n0, n=n, nc=nc,
                theta=_theta(p) if theta is None else theta, g=g, search=search, nrays=nrays,
                precision=precision, response=response, stages=stages)


def _theta(p):
    """A lengthscale for uniform designs in p inputs, through the workloads'
    settings (0.1 in 2-d, 0.25 in 4-d, 1 in 8-d)."""
    return round(0.05 * 1.45 ** p, 4)


def listed():
    return [
        # an online request for one location against a resident design: the
        # smallest call, all latency
        _case("serve_1_ray_8d", "serve", 1_000_000, 8, 1, 50, 1000, nrays=8, theta=1.0),
        # a small dense 2-d problem in the parity arithmetic (a first try, a
        # regression check)
        _case("dense_2d_exh_fp64", "predict", 4000, 2, 100, 30, 500, "exhaustive",
              precision="fp64", theta=0.1),
        # the headline workload: a million 8-d points, 100,000 locations, rays
        _case("ray_8d", "predict", 1_000_000, 8, 100_000, 50, 1000, nrays=8, theta=1.0),
        # the same design, exhaustive search of a smaller batch
        _case("exh_8d", "predict", 1_000_000, 8, 20_000, 50, 1000, "exhaustive", theta=1.0),
        # the same through the tensor-core scorer
        _case("exh_tc_8d", "predict", 1_000_000, 8, 10_000, 50, 1000, "exhaustive",
              precision="fp32_tc", theta=1.0),
        # ray search with picks from the whole design, not only the candidates
        _case("ray_full_8d", "predict", 1_000_000, 8, 10_000, 50, 1000, "ray_full", nrays=8,
              theta=1.0),
        # the ill-conditioned 4-d workload, which needs binary64: rays
        _case("ray_fp64_4d", "predict", 100_000, 4, 2000, 50, 1000, nrays=4, precision="fp64",
              theta=0.25),
        # and exhaustive search
        _case("exh_fp64_4d", "predict", 100_000, 4, 777, 50, 1000, "exhaustive",
              precision="fp64", theta=0.25),
        # uneven local designs (n 20..100, N' 300..2000) replayed as one graph:
        # a nightly batch with per-location budgets
        _case("uneven_plan_ray_8d", "plan", 1_000_000, 8, 10_000, 100, 2000, nrays=8, theta=1.0),
        # the gridded 2-d experiment, two stages of local inference for theta,
        # one ray, an odd number of locations
        _case("two_stage_mle_2d", "mle", 40_401, 2, 9801, 50, 1000, nrays=1, theta=0.5,
              response="grid"),
        # global separable lengthscales on 1,000 rows (the pre-scaling fit)
        _case("prescale_fit_8d", "fit", 100_000, 8, 1, 1000, 1000, theta=1.0),
        # candidates alone, for a caller with its own local model: a small 3-d
        # design with many neighbours (the whole design is streamed)
        _case("knn_3d_N37908", "knn", 37_908, 3, 5001, 1, 2000),
    ]


def draw(rng):
    """One more case from the ranges the listed ones stand for."""
    def lu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["predict"] * 6 + ["serve", "plan", "mle", "fit", "knn", "knn"])
    p = rng.randint(2, 10)
    N = lu(4000, 1_000_000)
    if kind == "fit":
        return _drop(_case("", "fit", N, p, 1, rng.randint(100, 1000), 1000))
    nc = min(rng.randint(200, 2000), N // 2)
    if kind == "knn":
        return _drop(_case("", "knn", N, p, lu(1, 20_000), 1, nc))
    n = rng.randint(15, 100 if kind != "mle" else 64)
    search = rng.choice(["ray", "ray", "exhaustive", "ray_full"])
    precision = rng.choice(["fp32", "fp32", "fp32_tc", "fp64", "fp32_promote"])
    # binary64 scoring is the slow parity arithmetic: fewer locations
    M = lu(1, 150 if precision in ("fp64", "fp32_promote") else 10_000)
    if kind == "serve":
        search, precision, M = "ray", "fp32", lu(1, 2000)
    elif kind == "mle":
        search, M = rng.choice(["ray", "exhaustive"]), min(M, 5000)
    elif kind == "plan":
        precision, n, nc = "fp32", max(n, 30), max(nc, 300)
    return _drop(_case("", kind, N, p, M, n, nc, search, rng.randint(1, p), precision,
                       n0=rng.choice([4, 6, 10])))


def _drop(c):
    del c["name"]
    return c


# ----- inputs -------------------------------------------------------------------------


def _w2(x):
    return torch.exp(-(x - 1) ** 2) + torch.exp(-0.8 * (x + 1) ** 2) - 0.05 * torch.sin(8 * (x + 0.1))


def _inputs(c, seed):
    """Design, responses and locations (binary64, on the GPU) from the seed."""
    gen = torch.Generator(device=DEV).manual_seed(seed)

    def rand(*shape):
        return torch.rand(shape, generator=gen, device=DEV, dtype=torch.float64)

    N, p, M = c["N"], c["p"], c["M"]
    if c["response"] == "grid":
        side = math.isqrt(N)
        ax = torch.linspace(-2, 2, side, device=DEV, dtype=torch.float64)
        X = torch.cartesian_prod(ax, ax).contiguous()
        xr = 3.96 * rand(M, p) - 1.98
        y = -_w2(X[:, 0]) * _w2(X[:, 1])
    else:
        X, a, phi, xr = rand(N, p), 0.5 + 1.5 * rand(p), 2 * math.pi * rand(p), rand(M, p)
        y = torch.sin(2 * math.pi * a * X + phi).sum(1) + 0.3 * X.prod(1)
    n_loc = nc_loc = None
    if c["kind"] == "plan":
        n_loc = (20 + (rand(M) * (c["n"] - 19)).int()).clamp(max=c["n"]).int()
        nc_loc = (300 + (rand(M) * (c["nc"] - 299)).int()).clamp(max=c["nc"]).int()
    subset = None
    if c["kind"] == "fit":
        subset = torch.randperm(N, generator=gen, device=DEV)[: c["n"]].int()
    return X, y, xr, n_loc, nc_loc, subset


T_RANGE = (1e-3, 10.0)       # local lengthscales
FIT_RANGE = (1e-3, 1e3)      # global lengthscales


def prepare(case, seed):
    c = case
    X, y, xr, n_loc, nc_loc, subset = _inputs(c, seed)
    N, p, M, n, nc = c["N"], c["p"], c["M"], c["n"], c["nc"]
    search, prec = lagp.SEARCH[c["search"]], lagp.PRECISION[c["precision"]]
    s = dict(c=c, X=X, y=y, xr=xr, search=search, prec=prec)

    def dev(*shape, dtype=torch.float64):
        return torch.empty(shape, dtype=dtype, device=DEV)

    kind = c["kind"]
    if kind == "fit":
        s.update(subset=subset, theta=dev(p), info=dev(3, dtype=torch.int32),
                 ws=dev(lagp.laGP_sep_mle_workspace_bytes(n, p), dtype=torch.uint8))
        return s
    if kind == "knn":
        s.update(cand=dev(M, nc, dtype=torch.int32),
                 ws=dev(lagp.laGP_knn_workspace_bytes(N, p, M, nc), dtype=torch.uint8))
        return s
    shape = (N, p, M, n, nc, c["nrays"], search, prec)
    if kind == "serve":
        lib = lagp.load()
        need = lib.laGP_ctx_design_bytes(N, p) + lib.laGP_ctx_request_bytes(*shape, 0)
        s["ctx"] = lagp.Context(X, y, c["theta"], c["g"], c["n0"], nc, search, c["nrays"], prec,
                                need + (1 << 20), max_inflight=2)
        for k, t in (("hx", xr), ("hm", torch.empty(M)), ("hs", torch.empty(M))):
            s[k] = t.to("cpu", torch.float64).pin_memory().numpy()
        return s
    s.update(mean=dev(M), s2=dev(M))
    if kind == "mle":
        s.update(theta=dev(M), ws=dev(lagp.laGP_mle_workspace_bytes(*shape), dtype=torch.uint8))
        return s
    s["ws"] = dev(lagp.laGP_workspace_bytes(*shape), dtype=torch.uint8)
    if kind == "plan":
        s["plan"] = lagp.Plan(X, y, xr, c["n0"], n, nc, c["theta"], c["g"], search, c["nrays"],
                              prec, s["mean"], s["s2"], s["ws"], n_loc=n_loc, nclose_loc=nc_loc)
    return s


def run(state):
    s, c = state, state["c"]
    kind = c["kind"]
    if kind == "predict":
        lagp.laGP_build_and_predict(s["X"], s["y"], s["xr"], c["n0"], c["n"], c["nc"], c["theta"],
                                    c["g"], s["search"], c["nrays"], s["prec"], s["mean"], s["s2"],
                                    s["ws"])
        return dict(mean=s["mean"], s2=s["s2"])
    if kind == "plan":
        s["plan"].launch()
        return dict(mean=s["mean"], s2=s["s2"])
    if kind == "serve":
        s["ctx"].wait(s["ctx"].submit(s["hx"], c["n"], s["hm"], s["hs"]))
        return dict(mean=s["hm"], s2=s["hs"])
    if kind == "knn":
        lagp.laGP_knn(s["X"], s["xr"], c["nc"], s["cand"], s["ws"])
        return dict(cand=s["cand"])
    if kind == "mle":
        lagp.laGP_build_and_predict_mle(s["X"], s["y"], s["xr"], c["n0"], c["n"], c["nc"],
                                        c["theta"], c["g"], *T_RANGE, c["stages"], s["search"],
                                        c["nrays"], s["prec"], s["theta"], s["mean"], s["s2"],
                                        s["ws"])
        return dict(theta=s["theta"], mean=s["mean"], s2=s["s2"])
    lagp.laGP_sep_mle(s["X"], s["y"], s["subset"], c["g"], c["theta"], *FIT_RANGE, 200, s["theta"],
                      s["ws"], info=s["info"])
    return dict(theta=s["theta"])


def work(case):
    """Inputs read once and outputs written once; the method's operations:
    distances to the whole design, per greedy step the ALC evaluations through
    the factor (rays: 20 per ray, the usual length of a line search, and the
    snap), and the factor's growth."""
    c = case
    N, p, M, n0, n, nc = (c[k] for k in ("N", "p", "M", "n0", "n", "nc"))
    if c["kind"] == "fit":
        # at least 10 likelihood evaluations of one inversion each
        return dict(bytes=8 * n * (p + 1), flops=10 * 2.0 * n ** 3)
    nbytes, flops = 8 * (N * p + M * p), 3.0 * N * p * M
    if c["kind"] == "knn":
        return dict(bytes=nbytes + 4 * M * nc, flops=flops)
    if c["kind"] == "plan":                      # the average location
        n, nc = (20 + n) // 2, (300 + nc) // 2
    R = c["nrays"] or p
    steps = range(n0, n)
    if c["search"] == "exhaustive":
        per = nc * (3 * p * n + sum(2 * j + 5 for j in steps))
    else:
        per = sum(20 * R * (j * j + (3 * p + 4) * j) + 3 * p * nc for j in steps)
    per += sum(4 * j * j + 3 * p * j for j in range(n))
    stages = c["stages"] if c["kind"] == "mle" else 1
    if c["kind"] == "mle":
        per += 4 * 3 * n ** 3                    # four likelihood evaluations a stage
    return dict(bytes=nbytes + 8 * N + 16 * M, flops=flops + M * stages * float(per))


# ----- the same results in plain torch, 64 bits -------------------------------------------


def _knn(X, xr, nc):
    out = []
    rows = max(1, (1 << 27) // X.shape[0])
    for x in xr.split(rows):
        d = torch.zeros(x.shape[0], X.shape[0], dtype=torch.float64, device=X.device)
        for k in range(X.shape[1]):
            d += (X[:, k][None, :] - x[:, k, None]) ** 2
        out.append(d.topk(nc, largest=False, sorted=True).indices)
    return torch.cat(out)


def _corr(a, b, theta):
    """exp(-|a - b|^2 / theta): a [m][i][p], b [m][j][p], theta [m]."""
    return torch.exp(-((a[:, :, None] - b[:, None]) ** 2).sum(-1) / theta[:, None, None])


class _Design:
    """Local designs of m locations, grown one point at a time: L is the
    Cholesky factor of K_j, z = L^{-1} k(x), b = L^{-1} y."""

    def __init__(self, C, Cy, x, theta, n, g):
        m, nc, p = C.shape
        self.C, self.Cy, self.x, self.theta, self.g, self.j = C, Cy, x, theta, g, 0
        self.S = C.new_zeros(m, n, p)
        self.Sy = C.new_zeros(m, n)
        self.L = C.new_zeros(m, n, n)
        self.z, self.b = C.new_zeros(m, n), C.new_zeros(m, n)
        self.used = torch.zeros(m, nc, dtype=torch.bool, device=C.device)
        self.kx = _corr(C, x[:, None], theta)[:, :, 0]
        self.ar = torch.arange(m, device=C.device)

    def w(self, Z):
        """L^{-1} K(S, Z) [m][j][points]."""
        j = self.j
        return torch.linalg.solve_triangular(self.L[:, :j, :j],
                                             _corr(self.S[:, :j], Z, self.theta), upper=False)

    def add(self, r):
        j = self.j
        s, sy = self.C[self.ar, r], self.Cy[self.ar, r]
        ks = self.kx[self.ar, r]
        if j:
            l = self.w(s[:, None])[:, :, 0]
            self.L[:, j, :j] = l
            v = 1 + self.g - (l * l).sum(1)
            ks = ks - (l * self.z[:, :j]).sum(1)
            t = sy - (l * self.b[:, :j]).sum(1)
        else:
            l, v, t = None, torch.full_like(ks, 1 + self.g), sy
        d = v.sqrt()
        self.L[:, j, j] = d
        self.z[:, j], self.b[:, j] = ks / d, t / d
        self.S[:, j], self.Sy[:, j] = s, sy
        self.used[self.ar, r] = True
        self.j += 1
        return l, d, self.z[:, j]

    def alc(self, Z):
        w = self.w(Z)
        num = torch.einsum("mjr,mj->mr", w, self.z[:, : self.j]) - \
            _corr(Z, self.x[:, None], self.theta)[:, :, 0]
        v = 1 + self.g - (w * w).sum(1)
        return torch.where(v > 0, num * num / v, 0.0)

    def predict(self):
        j = self.j
        mean = (self.z * self.b).sum(1)
        s2 = (self.b ** 2).sum(1) * (1 + self.g - (self.z ** 2).sum(1)) / j
        return mean, s2


def _exhaustive(D, n0, n):
    m, nc, _ = D.C.shape
    W = D.C.new_zeros(m, nc, n)
    vs, ns = D.C.new_zeros(m, nc), D.C.new_zeros(m, nc)
    for j in range(n):
        if j < n0:
            r = torch.full((m,), j, device=D.C.device)
        else:
            v = 1 + D.g - vs
            alc = torch.where(v > 0, (ns - D.kx) ** 2 / v, 0.0).masked_fill(D.used, -1.0)
            r = alc.argmax(1)
        l, d, zj = D.add(r)
        k = _corr(D.C, D.S[:, j: j + 1], D.theta)[:, :, 0]
        if j:
            k = k - torch.bmm(W[:, :, :j], l[:, :, None])[:, :, 0]
        W[:, :, j] = k / d[:, None]
        vs += W[:, :, j] ** 2
        ns += W[:, :, j] * zj[:, None]


def _brent(f, shape, like):
    """Brent's (1973) bounded minimiser on [0, 1] for many functions at once."""
    tol3, eps, gold = 2.0 ** -13 / 3, 2.0 ** -26, (3 - math.sqrt(5)) / 2
    a, b = like.new_zeros(shape), like.new_ones(shape)
    x = like.new_full(shape, gold)
    w, v, d, e = x.clone(), x.clone(), a.clone(), a.clone()
    fx = f(x)
    fw, fv = fx.clone(), fx.clone()
    for _ in range(200):
        mid = (a + b) / 2
        t1 = eps * x.abs() + tol3
        live = (x - mid).abs() > 2 * t1 - (b - a) / 2
        if not bool(live.any()):
            break
        r, q = (x - w) * (fx - fv), (x - v) * (fx - fw)
        pn, q = (x - v) * q - (x - w) * r, 2 * (q - r)
        pn, q = torch.where(q > 0, -pn, pn), q.abs()
        tryp = e.abs() > t1
        par = tryp & (pn.abs() < (q * e / 2).abs()) & (pn > q * (a - x)) & (pn < q * (b - x))
        dp = pn / torch.where(par, q, 1.0)
        u = x + dp
        edge = (u - a < 2 * t1) | (b - u < 2 * t1)
        dp = torch.where(edge, torch.where(mid >= x, t1, -t1), dp)
        eg = torch.where(x < mid, b - x, a - x)
        e = torch.where(live, torch.where(par, d, eg), e)
        d = torch.where(live, torch.where(par, dp, gold * eg), d)
        u = x + torch.where(d.abs() >= t1, d, torch.where(d >= 0, t1, -t1))
        fu = f(u)
        good = live & (fu <= fx)
        bad = live & ~good
        low = u < x
        a2 = torch.where(good & ~low, x, torch.where(bad & low, u, a))
        b = torch.where(good & low, x, torch.where(bad & ~low, u, b))
        a = a2
        sec = bad & ((fu <= fw) | (w == x))
        thi = bad & ~sec & ((fu <= fv) | (v == x) | (v == w))
        v = torch.where(good | sec, w, torch.where(thi, u, v))
        fv = torch.where(good | sec, fw, torch.where(thi, fu, fv))
        w = torch.where(good, x, torch.where(sec, u, w))
        fw = torch.where(good, fx, torch.where(sec, fu, fw))
        x, fx = torch.where(good, u, x), torch.where(good, fu, fx)
    return x, fx


def _ray(D, n0, n, R, lo, hi):
    m, nc, p = D.C.shape
    rank = torch.arange(nc, device=D.C.device).expand(m, nc)
    for j in range(n):
        if j < n0:
            D.add(torch.full((m,), j, device=D.C.device))
            continue
        t = j - n0 + 1
        order = torch.where(D.used, nc, rank).sort(1).values       # unselected ranks first
        pos = (t % math.isqrt(t) + torch.arange(R, device=D.C.device)) % (nc - j)
        starts = order[:, pos]
        A = D.C.gather(1, starts[:, :, None].expand(m, R, p))
        dk = 10 * (A - D.x[:, None])
        face = torch.where(dk > 0, (hi - A) / dk, torch.where(dk < 0, (lo - A) / dk, 1.0))
        dk = dk * face.clamp(0, 1).amin(2, keepdim=True)
        s, fs = _brent(lambda u: -D.alc(A + u[:, :, None] * dk), (m, R), D.C)
        a0 = D.alc(A)
        stay = (a0 >= -fs) | ((dk * dk).sum(2) == 0)
        s, val = torch.where(stay, 0.0, s), torch.where(stay, a0, -fs)
        ib = val.argmax(1)
        xs = A[D.ar, ib] + s[D.ar, ib][:, None] * dk[D.ar, ib]
        dist = ((D.C - xs[:, None]) ** 2).sum(2)
        isstart = torch.zeros_like(D.used).scatter_(1, starts, True)
        free = ~D.used & (~isstart | (dist == 0))
        free = torch.where(free.any(1, keepdim=True), free, ~D.used)
        D.add(dist.masked_fill(~free, math.inf).argmin(1))


def _theta_hat(D, theta, tmin, tmax):
    """Maximiser of the marginal likelihood of each design: Newton's method
    kept inside a bracket from the sign of the derivative."""
    n, S, y = D.j, D.S[:, : D.j], D.Sy[:, : D.j, None]
    d2 = ((S[:, :, None] - S[:, None]) ** 2).sum(-1)
    eye = torch.eye(n, dtype=torch.float64, device=S.device)
    t = theta.clamp(tmin, tmax)
    lo, hi = torch.full_like(t, tmin), torch.full_like(t, tmax)
    run_ = torch.ones_like(t, dtype=torch.bool)
    for _ in range(200):
        tt = t[:, None, None]
        K = torch.exp(-d2 / tt) * (1 - eye)
        K1 = K * d2 / tt ** 2
        K2 = K1 * (d2 / tt ** 2 - 2 / tt)
        Ki = torch.linalg.inv(K + (1 + D.g) * eye)
        al = Ki @ y
        G, u = Ki @ K1, K1 @ al

        def tr(a, b):
            return (a * b.transpose(1, 2)).sum((1, 2))

        psi = (y * al).sum((1, 2))
        p1, p2 = -(al * u).sum((1, 2)), 2 * (u * (Ki @ u)).sum((1, 2)) - (al * (K2 @ al)).sum((1, 2))
        g1 = -0.5 * tr(Ki, K1) - n / 2 * p1 / psi
        g2 = -0.5 * (tr(Ki, K2) - tr(G, G)) - n / 2 * (p2 / psi - (p1 / psi) ** 2)
        lo, hi = torch.where(run_ & (g1 > 0), t, lo), torch.where(run_ & (g1 <= 0), t, hi)
        tn = t - g1 / g2
        tn = torch.where((g2 < 0) & (tn > lo) & (tn < hi), tn, (lo + hi) / 2)
        stop = (hi - lo) <= 1e-10 * t
        tn = torch.where(run_ & ~stop, tn, t)
        run_ = run_ & ~stop & ((tn - t).abs() > 1e-10 * tn)
        t = tn
        if not bool(run_.any()):
            break
    return t


def _exact_fit(c, X, y, subset):
    S, ys = X[subset.long()], y[subset.long()]
    n, p = S.shape
    d2 = (S[:, None] - S[None]) ** 2
    eye = torch.eye(n, dtype=torch.float64, device=S.device)
    lo, hi = math.log(FIT_RANGE[0]), math.log(FIT_RANGE[1])
    e = torch.full((p,), math.log(c["theta"]), dtype=torch.float64, device=S.device)

    def value(e):
        K = torch.exp(-(d2 @ torch.exp(-e))) * (1 - eye) + (1 + c["g"]) * eye
        L = torch.linalg.cholesky(K)
        a = torch.linalg.solve_triangular(L, ys[:, None], upper=False)
        return L.diagonal().log().sum() + n / 2 * torch.log((a * a).sum())

    e.requires_grad_(True)
    opt = torch.optim.LBFGS([e], max_iter=300, tolerance_grad=1e-9, tolerance_change=1e-13,
                            history_size=30, line_search_fn="strong_wolfe")

    def closure():
        opt.zero_grad()
        v = value(e)
        v.backward()
        return v

    opt.step(closure)
    e = e.detach()
    return None if bool(((e < lo + 1) | (e > hi - 1)).any()) else torch.exp(e)


def exact(case, seed):
    """Which points a design takes is decided by comparisons: exhaustive scores
    and binary64 rays make nearly the choices of this code, while the end of
    an FP32 line search, snapped to a candidate, has no value that another
    rounding would give.  s2 has none either: it is a difference of the order
    of the nugget, of designs that differ at near-ties."""
    c = case
    if c["search"] == "ray" and c["precision"] != "fp64" and c["kind"] in ("predict", "serve"):
        return None
    big = c["M"] * c["N"] > 3e10 or c["M"] * c["n"] ** 2 * c["nc"] > 1e11
    if c["kind"] in ("knn", "plan") or c["search"] == "ray_full" or (big and c["kind"] != "fit"):
        return None              # whole numbers, per-location sizes, or over 20 seconds
    X, y, xr, _, _, subset = _inputs(c, seed)
    if c["kind"] == "fit":
        th = _exact_fit(c, X, y, subset)
        return None if th is None else dict(theta=th)
    lo, hi = X.amin(0), X.amax(0)
    R = c["nrays"] or c["p"]
    parts = []
    for x in xr.split(max(1, (1 << 28) // (c["nc"] * c["n"]))):
        cand = _knn(X, x, c["nc"])
        C, Cy = X[cand], y[cand]

        def design(theta):
            D = _Design(C, Cy, x, theta, c["n"], c["g"])
            if c["search"] == "exhaustive":
                _exhaustive(D, c["n0"], c["n"])
            else:
                _ray(D, c["n0"], c["n"], R, lo, hi)
            return D

        theta = torch.full((x.shape[0],), c["theta"], dtype=torch.float64, device=DEV)
        if c["kind"] != "mle":
            parts.append(design(theta).predict())
            continue
        D = None
        for _ in range(c["stages"]):
            D = design(theta)
            theta = _theta_hat(D, theta, *T_RANGE)
        F = _Design(C, Cy, x, theta, c["n"], c["g"])   # the last design at its own estimate
        F.C, F.Cy, F.kx = D.S, D.Sy, _corr(D.S, x[:, None], theta)[:, :, 0]
        F.used = torch.zeros(D.S.shape[:2], dtype=torch.bool, device=DEV)
        for j in range(c["n"]):
            F.add(torch.full((x.shape[0],), j, device=DEV))
        parts.append((theta,) + F.predict())
    names = ("theta", "mean", "s2") if c["kind"] == "mle" else ("mean", "s2")
    return {**{k: torch.cat(v) for k, v in zip(names, zip(*parts))}, "s2": None}
