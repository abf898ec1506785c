"""The calls that a user of this library makes, at the sizes they make them, as timed cases.

Each case goes through a public entry point (``Context`` or the C ABI of ``include/gp2s.h``) on
seeded synthetic inputs of the shapes in ``paper_2512_06143_gb300/workloads.py``: clustered 3-D
points, the sphere x time x elevation set, uniform points in 1 to 3 dimensions.  Options are the
library's defaults unless a case says otherwise, so a second evaluation on the same points reuses
the pattern as a training loop does.  ``exact`` restates the same quantities in FP64 with plain torch
(neighbour pairs, conjugate gradients, Lanczos quadrature with the same probes, autograd).
"""
import ctypes
import math

import numpy as np
import torch

import paper_2512_06143_gb300 as gp

DEV = "cuda"


def listed():
    """`layout` fixes where clusters and bumps lie; the points, the noise and the probes' pairing with
    them come from the seed."""
    cases = [
        # the smallest call: a few hundred points, asynchronous, nothing allocated (a serving process or
        # a captured graph that owns the device's memory)
        dict(name="noalloc_2d_301", kind="noalloc", shape="uniform", n=301, d=2, row=30.0, L=3, sigma2=1e-3),
        # block-MCMC training on the paper's 1-D function (2,000 points): many small evaluations, launches
        # and the dense Cholesky count
        dict(name="mcmc_1d_2000", kind="mcmc", shape="f1", n=2000, d=1, row=80.0, L=2, sigma2=1e-4, iters=3),
        # the plain FP64 evaluation with the exact log-determinant (4,096 points in 2-D)
        dict(name="lml_exact_fp64_2d_4096", kind="lml", shape="uniform", n=4096, d=2, row=32.0, L=4, sigma2=1e-4,
             precision="fp64", logdet="exact", probes=64),
        # uneven independent problems in one call, 16 probes each (per-region or per-tenant models)
        dict(name="batch_24", kind="batch", shape="uniform", count=24, n=65536, n_min=2048, L=4, sigma2=1e-4, probes=16),
        # the log-determinant alone on a matrix that is already assembled, ragged size, 2-D
        dict(name="logdet_2d_200003", kind="logdet", shape="uniform", n=200003, d=2, row=60.0, L=4, sigma2=4e-4,
             probes=64),
        # one solve A a = y on an assembled matrix (a new response on the same points)
        dict(name="solve_3d_400001", kind="solve", shape="clusters", n=400001, d=3, row=100.0, L=8, sigma2=4e-4),
        # serving: posterior mean and variance at 200 test points of a 100,000-point model
        dict(name="posterior_3d_100000", kind="posterior", shape="clusters", n=100000, d=3, row=80.0, L=8, sigma2=4e-4,
             tests=200),
        # covariance assembly alone, pattern rebuilt, at the clustered benchmark's size
        dict(name="assemble_3d_1m", kind="assemble", shape="clusters", n=1000000, d=3, row=100.0, L=8, sigma2=4e-4),
        # LML + gradient with the convolution kernel's length-scale field, 32 probes
        dict(name="grad_wendconv_2d_100003", kind="grad", shape="uniform", family="wendconv", n=100003, d=2, row=40.0, L=3,
             sigma2=1e-3, probes=32),
        # LML + gradient in plain FP64 (no mixed precision), 16 probes
        dict(name="grad_fp64_3d_30011", kind="grad", shape="uniform", n=30011, d=3, row=50.0, L=4, sigma2=1e-3,
             precision="fp64", probes=16),
        # the training step of the 1M-point benchmark: LML + 42-parameter gradient, 64 probes
        dict(name="grad_clusters_3d_1m", kind="grad", shape="clusters", n=1000000, d=3, row=100.0, L=8, sigma2=4e-4,
             probes=64),
        # the same on the sphere x time x elevation set of the 10M-point workload, 8M points, 32 probes
        dict(name="grad_sphere_4d_8m", kind="grad", shape="sphere", n=8000000, d=4, row=60.0, L=8, sigma2=4e-4,
             probes=32),
    ]
    return [dict(c, layout=3) for c in cases]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    return dict(_draw(rng), layout=rng.randint(0, 1000))


def _draw(rng):
    kind = rng.choice(["noalloc", "mcmc", "lml", "batch", "logdet", "solve", "posterior", "assemble", "wendconv", "fp64",
                       "clusters", "sphere"])
    d = rng.randint(1, 3)
    row = float(_log(rng, 20, 150))
    if kind == "noalloc":
        n = _log(rng, 16, 512)
        return dict(kind=kind, shape="uniform", n=n, d=d, row=min(30.0, n / 4), L=rng.randint(1, 6), sigma2=1e-3)
    if kind == "mcmc":
        return dict(kind=kind, shape="f1", n=_log(rng, 500, 4000), d=1, row=80.0, L=2, sigma2=1e-4, iters=rng.randint(1, 3))
    if kind == "lml":
        return dict(kind=kind, shape="uniform", n=_log(rng, 1000, 8000), d=d, row=min(row, 60.0), L=4, sigma2=1e-4,
                    precision=rng.choice(["fp64", "mixed"]), logdet="exact", probes=64)
    if kind == "batch":
        return dict(kind=kind, shape="uniform", count=rng.randint(6, 24), n=_log(rng, 8192, 65536), n_min=2048, L=4,
                    sigma2=1e-4, probes=16)
    if kind == "logdet":
        return dict(kind=kind, shape=rng.choice(["uniform", "clusters"]), n=_log(rng, 25000, 400000), d=max(2, d), row=row,
                    L=rng.randint(2, 8), sigma2=4e-4, probes=rng.choice([16, 32, 48, 64]))
    if kind == "solve":
        return dict(kind=kind, shape="clusters", n=_log(rng, 30000, 600000), d=max(2, d), row=row, L=8, sigma2=4e-4)
    if kind == "posterior":
        return dict(kind=kind, shape="clusters", n=_log(rng, 20000, 200000), d=max(2, d), row=row, L=8, sigma2=4e-4,
                    tests=_log(rng, 16, 256))
    if kind == "assemble":
        return dict(kind=kind, shape=rng.choice(["uniform", "clusters", "sphere"]), n=_log(rng, 20000, 2000000), d=d, row=row,
                    L=8, sigma2=4e-4)
    if kind == "wendconv":
        return dict(kind="grad", shape="uniform", family="wendconv", n=_log(rng, 25000, 150000), d=max(2, d), row=40.0,
                    L=rng.randint(2, 4), sigma2=1e-3, probes=rng.choice([16, 32, 64]))
    if kind == "fp64":
        return dict(kind="grad", shape="uniform", n=_log(rng, 21000, 50000), d=max(2, d), row=50.0, L=4, sigma2=1e-3,
                    precision="fp64", probes=16)
    if kind == "clusters":
        return dict(kind="grad", shape="clusters", n=_log(rng, 50000, 1000000), d=3, row=100.0, L=8, sigma2=4e-4,
                    probes=rng.choice([32, 64]))
    return dict(kind="grad", shape="sphere", n=_log(rng, 200000, 7000000), d=4, row=60.0, L=8, sigma2=4e-4, probes=32)


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _points(case, n, d, g, lay):
    """n points in [0, 1]^d and their observations, FP64 on the GPU.  `lay` draws what belongs to the
    place and not to the sample: cluster centers, the elevation field."""
    def u(*s):
        return torch.rand(*s, generator=g, device=DEV, dtype=torch.float64)

    def z(*s):
        return torch.randn(*s, generator=g, device=DEV, dtype=torch.float64)
    shape = case["shape"]
    if shape == "f1":
        X = u(n, 1).sort(0).values
        x = X[:, 0]
        return X, torch.sin(5 * x) + torch.cos(20 * x) + 2 * (x - 0.4) ** 2 * torch.cos(400 * x) + 0.01 * z(n)
    if shape == "sphere":
        lon, t = u(n) * (2 * math.pi), u(n)
        lat = torch.asin(u(n) * 2 - 1)
        e = torch.zeros_like(lon)
        for _ in range(16):
            kx, ky = lay.integers(1, 6, 2)
            ph = lay.random(2) * 2 * math.pi
            amp = float(lay.normal()) / float(kx + ky)
            e += amp * torch.sin(float(kx) * lon + ph[0]) * torch.cos(float(ky) * lat + ph[1])
        e = (e - e.min()) / (e.max() - e.min())
        X = torch.stack([lon / (2 * math.pi), (lat + math.pi / 2) / math.pi, t, e], 1).contiguous()
        y = (torch.sin(2 * math.pi * X[:, 0]) * torch.cos(math.pi * X[:, 1]) + 0.5 * torch.sin(2 * math.pi * X[:, 2])
             + 0.5 * X[:, 3] + 0.02 * z(n))
        return X, y
    if shape == "clusters":
        lab = (u(n) * 50).long()
        X = (torch.tensor(lay.random((50, d)), device=DEV)[lab] + 0.03 * z(n, d)).clamp(0.0, 1.0)
    else:
        X = u(n, d)
    y = torch.sin(2 * math.pi * X[:, 0])
    if d > 1:
        y = y + torch.sin(4 * math.pi * X[:, 1] + 1.0)
    if d > 2:
        y = y + torch.sin(6 * math.pi * X[:, 2] + 2.0)
    return X, y + 0.02 * z(n)


def _radius(X, row, g):
    """Support radius whose mean number of stored entries per row is about `row` (counted on a sample)."""
    n, d = X.shape
    k = min(n, 256)
    sample = X[torch.randint(0, n, (k,), generator=g, device=DEV)]
    near = []
    for p in range(0, n, 1 << 20):
        d2 = torch.zeros(k, min(n - p, 1 << 20), device=DEV, dtype=torch.float64)
        for j in range(d):
            d2 += (sample[:, j, None] - X[None, p:p + (1 << 20), j]) ** 2
        near.append(torch.topk(d2.reshape(-1), min(d2.numel(), int(row * k) + 1), largest=False).values)
    near = torch.cat(near).sort().values
    return float("%.6g" % math.sqrt(float(near[min(len(near) - 1, int(row * k))])))


def _problem(case, seed, n, d, row, layout):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 17)
    rng = np.random.default_rng(layout)
    X, y = _points(case, n, d, g, rng)
    r = _radius(X, row, g)
    L = case["L"]
    if case.get("family") == "wendconv":
        h = gp.Hyper(d=d, r=r, sigma2=case["sigma2"], centers=rng.random((L, d)), radii=rng.uniform(0.3, 0.6, L),
                     amps=rng.uniform(0.2, 1.0, L), w0=1.0, family=gp.KERNEL_WENDCONV, ell=rng.uniform(0.7, 1.4, d),
                     G=rng.uniform(0.0, 1.5, (L, d)))
    else:
        h = gp.Hyper(d=d, r=r, sigma2=case["sigma2"], centers=rng.random((L, d)),
                     radii=np.full(L, 0.3 if case["shape"] == "sphere" else 0.4), amps=np.ones(L),
                     w0=1.0 if case["shape"] == "f1" else 0.0)
    return X, y, h


def _dim(case):
    return 4 if case["shape"] == "sphere" else case["d"]


def _batch_sizes(case):
    """(n, d, entries per row) of each problem of a batch: sizes spread over their logarithm, mixed dimensions."""
    k = case["count"]
    rng = np.random.default_rng(k)
    lo, hi = math.log(case["n_min"]), math.log(case["n"])
    return [(int(math.exp(lo + (hi - lo) * (b + 0.5) / k)), 1 + b % 3, float(math.exp(rng.uniform(math.log(10), math.log(200)))))
            for b in range(k)]


def _opts(case):
    kw = {}
    if case.get("precision") == "fp64":
        kw["precision"] = gp.PREC_FP64
    if case.get("logdet") == "exact":
        kw["logdet"] = gp.LOGDET_EXACT
    if case["kind"] == "logdet":
        kw["logdet"] = gp.LOGDET_SLQ
    if case["kind"] == "assemble":
        kw["pattern_cache"] = 1      # the pattern is rebuilt on every call
    if "probes" in case:
        kw["probes"] = case["probes"]
    return gp.default_opts(**kw)


def _mcmc_plan(case, seed, h):
    """Three blocks (centers; radii and amplitudes; noise), small steps, given random numbers."""
    P, L, d = h.nparams, h.L, h.d
    block = np.concatenate([np.zeros(L * d), np.ones(2 * L), [-1], [2]]).astype(np.int32)
    step = np.concatenate([np.full(L * d, 0.02), np.full(2 * L, 0.02), [0.0], [1e-6]])
    rng = np.random.default_rng(int(seed) + 31)
    lower = np.concatenate([np.full(L * d, -1.0), np.full(2 * L, 0.05), [0.0], [1e-7]])
    return dict(block=block, step=step, iters=case["iters"], lower=lower, upper=np.full(P, 10.0),
                normals=rng.standard_normal((case["iters"], P)), uniforms=rng.random((case["iters"], 3)))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        problems = [_problem(case, int(seed) * 64 + b, *s, case["layout"] + b) for b, s in enumerate(_batch_sizes(case))]
        return dict(case=case, ctx=gp.Context(0), problems=problems, opts=_opts(case))
    X, y, h = _problem(case, seed, case["n"], _dim(case), case["row"], case["layout"])
    s = dict(case=case, X=X, y=y, h=h)
    if kind == "noalloc":
        s["out"] = torch.empty(3, dtype=torch.float64, device=DEV)
        s["call"] = gp.load().gp2s_lml_exact_noalloc
        s["hc"] = h.c()
        return s
    s["ctx"], s["opts"] = gp.Context(0), _opts(case)
    if kind == "mcmc":
        s["plan"] = _mcmc_plan(case, seed, h)
    elif kind == "assemble":
        # the caller's own arrays: the matrix is handed on in buffers of one capacity for every seed
        cap = int(1.5 * case["n"] * case["row"]) + 4096
        s["buf"] = {k: torch.zeros(cap, dtype=t, device=DEV)
                    for k, t in (("col", torch.int32), ("val32", torch.float32), ("val64", torch.float64))}
    elif kind in ("logdet", "solve", "posterior"):
        s["ctx"].assemble(X, h, s["opts"])
        if kind == "posterior":
            s["ctx"].solve(y)
            s["Xs"] = X[:: max(1, case["n"] // case["tests"])][:case["tests"]] + 0.1 * h.r
    return s


def run(state):
    kind = state["case"]["kind"]
    if kind == "noalloc":
        st = state["call"](state["X"].shape[0], state["X"].data_ptr(), state["y"].data_ptr(), ctypes.byref(state["hc"]),
                           state["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if st != gp.OK:
            raise gp.GP2SError(st, "gp2s_lml_exact_noalloc")
        return state["out"]
    ctx = state["ctx"]
    if kind == "batch":
        return ctx.lml_batched(state["problems"], state["opts"])[0]
    X, y, h, opts = state["X"], state["y"], state["h"], state.get("opts")
    if kind == "mcmc":
        chain, accept, _ = ctx.mcmc(X, y, h, opts=opts, **state["plan"])
        return {"chain": chain, "accept": accept}
    if kind == "lml":
        return ctx.lml(X, y, h, opts)[0]
    if kind == "grad":
        lml, grad, _ = ctx.lml_grad(X, y, h, opts)
        return {"lml": lml, "grad": grad}
    if kind == "logdet":
        return ctx.logdet()[0]
    if kind == "solve":
        return ctx.solve(y)[0]
    if kind == "posterior":
        mean, var, _ = ctx.posterior(state["Xs"])
        return {"mean": mean, "var": var}
    ctx.assemble(X, h, opts)
    m = ctx.csr()
    for k, buf in state["buf"].items():
        buf[:m["nnz"]].copy_(m[k])
    return dict(state["buf"], rowptr=m["rowptr"], perm=m["perm"], dscale=m["dscale"])


def work(case):
    """The least one pass has to do: the points, observations and results once; an assembly writes its
    matrix once; a Krylov call multiplies by the matrix (FP32 or FP64 values, int32 columns) at least
    as often as its Lanczos steps (a solve: once), each input and output vector once per product; a
    dense factorisation is n^3 / 3 multiply-adds."""
    kind = case["kind"]
    steps = 100

    def one(n, d, row, m, grad=False):
        v = 8 if case.get("precision") == "fp64" else 4
        nnz = n * row
        b = steps * (nnz * (v + 4) + 2 * n * (m + 1) * v) + 8 * n * (d + 1)
        f = steps * 2 * nnz * (m + 1)
        return b, f + (4 * nnz * m if grad else 0)
    if kind == "batch":
        parts = [one(n, d, row, case["probes"]) for n, d, row in _batch_sizes(case)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    n, d, row = case["n"], _dim(case), case["row"]
    io = 8 * n * (d + 1)
    if kind == "noalloc":
        return {"bytes": io + 24, "flops": n ** 3 / 3}
    if kind == "mcmc":
        evals = 3 * case["iters"] + 1
        return {"bytes": io * evals, "flops": evals * n ** 3 / 3}
    if kind == "lml":
        return {"bytes": io + 8, "flops": n ** 3 / 3}
    if kind == "assemble":
        return {"bytes": 8 * n * d + n * row * 16 + 16 * n, "flops": n * row / 2 * (3 * d + 20 + 2 * case["L"])}
    if kind == "solve":
        return {"bytes": n * row * 8 + 16 * n, "flops": 2 * n * row}
    if kind == "posterior":
        m = case["tests"]
        return {"bytes": n * row * 8 + 8 * n * (d + 1) + 8 * m * (d + 2), "flops": 2 * n * row * m}
    b, f = one(n, d, row, case["probes"], kind == "grad")
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------------------
# the same quantities in FP64 with plain torch
# ---------------------------------------------------------------------------------------------
def _bumps(X, h, th):
    """Unscaled bump shapes on X: exp form (product kernel) or (1 - s)^3 (convolution kernel), n x L."""
    L, d = h.L, h.d
    c, rho = th[:L * d].reshape(L, d), th[L * d:L * d + L]
    s = ((X[:, None, :] - c[None]) ** 2).sum(2) / rho ** 2
    inside = s < 1.0
    s = torch.where(inside, s, torch.zeros_like(s))
    e = (1 - s) ** 3 if h.family == gp.KERNEL_WENDCONV else torch.exp(h.beta * (1 - 1 / (1 - s)))
    return torch.where(inside, e, torch.zeros_like(e))


def _taper(d, t):
    p = 4 if d <= 3 else 5
    return (1 - t).clamp(min=0.0) ** p * (p * t + 1)


def _fields(X, h, th):
    """Per-point factors: bump values times amplitudes (product kernel), or (signal, length scales)."""
    L, d = h.L, h.d
    e, amps = _bumps(X, h, th), th[L * d + L:L * d + 2 * L]
    if h.family != gp.KERNEL_WENDCONV:
        return (e * amps,)
    o = L * d + 2 * L
    G, ell, w0 = th[o:o + L * d].reshape(L, d), th[o + L * d:o + L * d + d], th[o + L * d + d]
    return w0 + e @ amps, ell ** 2 + e @ G


def _pair_values(X, h, th, i, j, f):
    """Kernel values of the pairs (i, j), i != j."""
    D2 = (X[i] - X[j]) ** 2
    if h.family != gp.KERNEL_WENDCONV:
        q = D2.sum(1)
        return _taper(h.d, torch.sqrt(q) / th[-2]) * ((f[0][i] * f[0][j]).sum(1) + h.w0)
    sig, lam = f
    m = (lam[i] + lam[j]) * 0.5
    pref = ((lam[i] * lam[j]) ** 0.25 / torch.sqrt(m)).prod(1)
    return sig[i] * sig[j] * pref * _taper(h.d, torch.sqrt((D2 / m).sum(1)) / th[-2])


def _diag(h, th, f):
    k = (f[0] ** 2).sum(1) + h.w0 if h.family != gp.KERNEL_WENDCONV else f[0] ** 2
    return k + th[-1]


def _cells(X, lo, edge):
    c = torch.floor((X - lo) / edge).long() + 1
    dims = c.max(0).values + 2
    key = c[:, 0]
    for k in range(1, X.shape[1]):
        key = key * dims[k] + c[:, k]
    return c, dims, key


def _pairs(X, reach, Y=None):
    """All (i, j) with |X_i - Y_j| < reach by a cell list; with Y None, the pairs i < j of X."""
    own = Y is None
    Y = X if own else Y
    n, d = X.shape
    lo = torch.minimum(X.min(0).values, Y.min(0).values)
    both = torch.cat([X, Y])
    c, dims, key = _cells(both, lo, reach * (1 + 1e-9))
    cx, ykey = c[:n], key[n:]
    order = torch.argsort(ykey)
    sk = ykey[order].contiguous()
    ii, jj = [], []
    for o in range(3 ** d):
        off = torch.tensor([(o // 3 ** k) % 3 - 1 for k in range(d)], device=DEV)
        cc = cx + off
        k = cc[:, 0]
        for a in range(1, d):
            k = k * dims[a] + cc[:, a]
        s, e = torch.searchsorted(sk, k), torch.searchsorted(sk, k, right=True)
        cnt = e - s
        for p in range(0, n, 1 << 18):
            q = cnt[p:p + (1 << 18)]
            i = torch.repeat_interleave(torch.arange(p, p + len(q), device=DEV), q)
            first = torch.repeat_interleave(torch.cumsum(q, 0) - q, q)
            j = order[s[i] + torch.arange(len(i), device=DEV) - first]
            keep = i < j if own else torch.ones_like(i, dtype=torch.bool)
            i, j = i[keep], j[keep]
            near = ((X[i] - Y[j]) ** 2).sum(1) < reach * reach
            ii.append(i[near])
            jj.append(j[near])
    return torch.cat(ii), torch.cat(jj)


class _Exact:
    """A = K + sigma^2 I of one problem in FP64, Jacobi-scaled (Ah = S A S)."""

    def __init__(self, X, h):
        self.X, self.h, self.n = X, h, X.shape[0]
        self.th = torch.tensor(h.theta(), device=DEV)
        f = _fields(X, h, self.th)
        reach = h.r
        if h.family == gp.KERNEL_WENDCONV:
            reach = h.r * math.sqrt(float(f[1].max())) * (1 + 1e-9)
        i, j = _pairs(X, reach)
        if h.family == gp.KERNEL_WENDCONV:
            q = ((X[i] - X[j]) ** 2 / ((f[1][i] + f[1][j]) * 0.5)).sum(1)
            i, j = i[q < h.r * h.r], j[q < h.r * h.r]
        self.i, self.j, self.f = i, j, f
        self.D = _diag(h, self.th, f)
        self.s = 1 / torch.sqrt(self.D)
        v = _pair_values(X, h, self.th, i, j, f) * (self.s[i] * self.s[j])
        k = torch.arange(self.n, device=DEV)
        self.Ah = torch.sparse_coo_tensor(torch.stack([torch.cat([i, j, k]), torch.cat([j, i, k])]),
                                          torch.cat([v, v, torch.ones(self.n, device=DEV, dtype=torch.float64)]),
                                          (self.n, self.n)).coalesce().to_sparse_csr()

    def cg(self, B, tol, keep=0, most=20000):
        """Ah^{-1} B by conjugate gradients, and the first `keep` step lengths and direction coefficients."""
        x, r, p = torch.zeros_like(B), B.clone(), B.clone()
        rho = (r * r).sum(0)
        b2 = rho.clone()
        rec = []
        for it in range(most):
            q = self.Ah @ p
            al = rho / (p * q).sum(0)
            al = torch.where(rho > 1e-30 * b2, al, torch.zeros_like(al))
            x += al * p
            r -= al * q
            new = (r * r).sum(0)
            be = torch.where(rho > 1e-30 * b2, new / rho, torch.zeros_like(new))
            if it < keep:
                rec.append((al, be))
            rho = new
            if it + 1 >= keep and it % 8 == 0 and bool((rho <= tol * tol * b2).all()):
                break
            p = r + be * p
        return x, rec

    def solve(self, y, tol=1e-13):
        """a = A^{-1} y, with one refinement of the residual."""
        b = (self.s * y)[:, None]
        x, _ = self.cg(b, tol)
        dx, _ = self.cg(b - self.Ah @ x, 1e-4)
        return self.s * (x + dx)[:, 0]

    def probes(self, m):
        """z_s[i] = 1 - 2 (top bit of splitmix64(s << 32 | i)), s = 1..m."""
        def wrap(c):
            return c - (1 << 64) if c >= 1 << 63 else c

        def shr(v, k):
            return (v >> k) & ((1 << (64 - k)) - 1)
        i = torch.arange(self.n, device=DEV)[:, None]
        v = (torch.arange(1, m + 1, device=DEV)[None] << 32) + i + wrap(0x9E3779B97F4A7C15)
        v = (v ^ shr(v, 30)) * wrap(0xBF58476D1CE4E5B9)
        v = (v ^ shr(v, 27)) * wrap(0x94D049BB133111EB)
        v = v ^ shr(v, 31)
        return torch.where(v < 0, -1.0, 1.0).double()

    def slq(self, rec):
        """log|A| from the recorded CG coefficients (the CG-Lanczos relation, Gauss quadrature)."""
        al, be = torch.stack([a for a, _ in rec]), torch.stack([b for _, b in rec])
        k = al.shape[0]
        dg = 1 / al
        dg[1:] += be[:-1] / al[:-1]
        off = torch.sqrt(be[:-1]) / al[:-1]
        T = torch.diag_embed(dg.T) + torch.diag_embed(off.T, 1) + torch.diag_embed(off.T, -1)
        w, V = torch.linalg.eigh(T[:, :k, :k].cpu())
        return float(torch.log(self.D).sum()) + self.n * float((V[:, 0, :] ** 2 * torch.log(w)).sum(1).mean())

    def lml(self, y, a, logdet):
        return -0.5 * float(y @ a) - 0.5 * logdet - 0.5 * self.n * math.log(2 * math.pi)

    def dense_logdet(self):
        L = torch.linalg.cholesky(self.Ah.to_dense())
        return float(torch.log(self.D).sum()) + 2 * float(torch.log(torch.diagonal(L)).sum())

    def grad(self, a, U, Z):
        """d LML / d theta from a = A^{-1} y and u = Ah^{-1} z: autograd of the kernel values at fixed weights."""
        U, V = self.s[:, None] * U, self.s[:, None] * Z
        m = U.shape[1]
        W = torch.empty(len(self.i), device=DEV, dtype=torch.float64)
        for p in range(0, len(W), 1 << 21):
            i, j = self.i[p:p + (1 << 21)], self.j[p:p + (1 << 21)]
            W[p:p + (1 << 21)] = a[i] * a[j] - ((U[i] * V[j]).sum(1) + (U[j] * V[i]).sum(1)) / (2 * m)
        Wd = a * a - (U * V).sum(1) / m
        th = self.th.clone().requires_grad_()
        f = _fields(self.X, self.h, th)
        ((_pair_values(self.X, self.h, th, self.i, self.j, f) * W).sum() + 0.5 * (_diag(self.h, th, f) * Wd).sum()).backward()
        return th.grad.cpu().numpy()


def _exact_lml(X, y, h, m, tol):
    E = _Exact(X, h)
    Z = E.probes(m)
    U, rec = E.cg(Z, tol, keep=100)
    a = E.solve(y)
    return E, a, Z, U, E.lml(y, a, E.slq(rec))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for b, s in enumerate(_batch_sizes(case)):
            X, y, h = _problem(case, int(seed) * 64 + b, *s, case["layout"] + b)
            out.append(_exact_lml(X, y, h, case["probes"], 1.0)[4])
        return np.array(out)
    if kind == "assemble" or case["n"] > 700000:
        return None     # the sorted numbering is the library's own; the largest gradients take too long
    X, y, h = _problem(case, seed, case["n"], _dim(case), case["row"], case["layout"])
    if kind == "grad":
        if case["n"] > 160000:
            return None
        E, a, Z, U, lml = _exact_lml(X, y, h, case["probes"], 1e-12)
        return {"lml": lml, "grad": E.grad(a, U, Z)}
    if kind == "mcmc":
        plan = _mcmc_plan(case, seed, h)

        def value(th):
            E = _Exact(X, h.with_theta(th))
            return E.lml(y, E.solve(y), E.dense_logdet())
        th, chain, accept = h.theta(), [], []
        v = value(th)
        for t in range(case["iters"]):
            took = []
            for b in range(3):
                new = np.where(plan["block"] == b, th + plan["step"] * plan["normals"][t], th)
                ok = bool((new >= plan["lower"]).all() and (new <= plan["upper"]).all())
                w = value(new) if ok else -math.inf
                took.append(int(ok and math.log(plan["uniforms"][t, b]) < w - v))
                if took[-1]:
                    th, v = new, w
            chain.append(np.concatenate([th, [v]]))
            accept.append(took)
        return {"chain": np.array(chain), "accept": np.array(accept, np.int32)}
    E = _Exact(X, h)
    if kind == "logdet":
        return E.slq(E.cg(E.probes(case["probes"]), 1.0, keep=100)[1])
    a = E.solve(y)
    if kind == "solve":
        return a
    if kind in ("noalloc", "lml"):
        ld = E.dense_logdet()
        lml = E.lml(y, a, ld)
        return torch.tensor([lml, float(y @ a), ld], dtype=torch.float64) if kind == "noalloc" else lml
    # posterior: k(x*, X) by the pairs between the test and training points
    Xs = X[:: max(1, case["n"] // case["tests"])][:case["tests"]] + 0.1 * h.r
    t, j = _pairs(Xs, h.r, X)
    fs = _fields(Xs, h, E.th)[0]
    v = _taper(h.d, torch.sqrt(((Xs[t] - X[j]) ** 2).sum(1)) / h.r) * ((fs[t] * E.f[0][j]).sum(1) + h.w0)
    K = torch.zeros(E.n, Xs.shape[0], device=DEV, dtype=torch.float64)
    K[j, t] = v
    B = E.s[:, None] * K
    x, _ = E.cg(B, 1e-11)
    return {"mean": K.T @ a, "var": (fs ** 2).sum(1) + h.w0 - (B * x).sum(0)}
