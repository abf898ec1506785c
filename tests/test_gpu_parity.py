"""CUDA path vs the FP64 oracle, element by element, through the C ABI (gp2s_* in libgp2s.so).

Tolerances:
  * pattern: identical sets of (row, column) pairs (bit-exact, FP64 support test on both sides);
  * FP64 values: max |dA| <= 1e-12 max |A|;
  * FP32 values (MIXED): max |dA| <= 1e-6 max |A| and |dA|_F <= 1e-6 |A|_F;
  * solve: |y - A_oracle a| / |y| <= 1e-8 with the oracle's FP64 A;
  * log-determinant: 1e-10 relative (exact path), 1e-3 relative with identical probes (SLQ);
  * gradient: Hutchinson with identical probes, max |dg| <= 1e-6 max |g|, in mixed precision (FP32
    probe solves to 1e-6) and in the FP64 form (solves to 1e-11).
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2512_06143_gb300 import workloads as W  # noqa: E402


@pytest.fixture(scope="module")
def gp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_06143_gb300 as gp
    from paper_2512_06143_gb300 import build
    build.build()
    gp.load()
    return gp


@pytest.fixture(scope="module")
def ctx(gp):
    return gp.Context(0)


def _csr_orig(c):
    """GPU CSR (sorted numbering) -> sorted arrays of original (row, col) keys and FP64 A values."""
    rp = c["rowptr"].cpu().numpy().astype(np.int64)
    col = c["col"].cpu().numpy().astype(np.int64)
    perm = c["perm"].cpu().numpy().astype(np.int64)
    s = c["dscale"].cpu().numpy()
    n = rp.shape[0] - 1
    rows = np.repeat(np.arange(n), np.diff(rp))
    A64 = c["val64"].cpu().numpy() / (s[rows] * s[col])
    A32 = None
    if c["val32"] is not None:
        A32 = c["val32"].cpu().numpy().astype(np.float64) / (s[rows] * s[col])
    key = perm[rows] * n + perm[col]
    order = np.argsort(key, kind="stable")
    return key[order], A64[order], (A32[order] if A32 is not None else None), rp, col


def _oracle_keys(csr):
    n = csr.n
    rows = np.repeat(np.arange(n), np.diff(csr.rowptr))
    return rows.astype(np.int64) * n + csr.col.astype(np.int64), csr.val


def _check_assembly(gp, ctx, w, exact_support=0, precision=None, method="auto"):
    import oracle
    h = gp.Hyper(**w["hyper"])
    opts = gp.default_opts(exact_support=exact_support)
    if precision is not None:
        opts.precision = precision
    X = torch.tensor(w["X"], dtype=torch.float64, device="cuda")
    info = ctx.assemble(X, h, opts)
    c = ctx.csr()
    key, A64, A32, rp, col = _csr_orig(c)
    ho = oracle.Hyper(**w["hyper"])
    ocsr = oracle.assemble(w["X"], ho, method)
    okey, oval = _oracle_keys(ocsr)
    assert info["nnz"] == ocsr.nnz
    assert np.array_equal(key, okey), "pattern differs from the oracle"
    amax = np.abs(oval).max()
    assert np.abs(A64 - oval).max() <= 1e-12 * amax
    if A32 is not None:
        d = A32 - oval
        assert np.abs(d).max() <= 1e-6 * amax
        assert np.linalg.norm(d) <= 1e-6 * np.linalg.norm(oval)
    # columns ascending within each sorted row, diagonal of Ah exactly 1
    n = rp.shape[0] - 1
    for i in range(0, n, max(1, n // 97)):
        cc = col[rp[i]:rp[i + 1]]
        assert np.all(np.diff(cc) > 0)
    v64 = c["val64"].cpu().numpy()
    rows = np.repeat(np.arange(n), np.diff(rp))
    assert np.all(v64[rows == col] == 1.0)
    # Ah is symmetric bit for bit, in FP64 and in its FP32 copy (each pair is evaluated once and
    # mirrored; the kernels are symmetric in their arithmetic anyway)
    import scipy.sparse as sp
    for v in (v64, None if c.get("val32") is None else c["val32"].cpu().numpy()):
        if v is None:
            continue
        S = sp.csr_matrix((v, col, rp), shape=(n, n))
        assert (S != S.T).nnz == 0
    return info


@pytest.mark.parametrize("d", [1, 2, 3, 4])
def test_assembly_random_dims(gp, ctx, d):
    w = W.random_small(100 + d, 6000 + 37 * d, d, L=3, clustered=(d % 2 == 1))
    _check_assembly(gp, ctx, w)


def test_assembly_paper_wendland_and_w0(gp, ctx):
    w = W.random_small(201, 5000, 3, L=2, kind=1, w0=0.5)
    _check_assembly(gp, ctx, w)


def test_assembly_small_2d_workload(gp, ctx):
    info = _check_assembly(gp, ctx, W.small_2d(0))
    assert 25 < info["nnz"] / info["n"] < 40


def test_assembly_guard_band_off_gives_identical_pattern(gp, ctx):
    w = W.random_small(202, 8000, 3, clustered=True)
    a = _check_assembly(gp, ctx, w, exact_support=0)
    b = _check_assembly(gp, ctx, w, exact_support=1)
    assert a["nnz"] == b["nnz"]
    assert b["band_pairs"] >= b["candidates"] - b["n"] - 1 or b["band_pairs"] > a["band_pairs"]


def test_assembly_fp64_precision(gp, ctx):
    w = W.random_small(203, 4000, 2)
    _check_assembly(gp, ctx, w, precision=gp.PREC_FP64)


def test_assembly_exact_boundary_grid(gp, ctx):
    # 2-D grid with spacing 1/8, r = 1/4: pairs at distance exactly r are excluded (strict <)
    g = np.arange(40) / 8.0
    X = np.array([[a, b] for a in g for b in g])
    w = dict(X=X, y=np.zeros(len(X)), hyper=dict(d=2, r=0.25, sigma2=1e-2, centers=np.array([[2.0, 2.0]]),
                                                  radii=np.array([3.0]), amps=np.array([1.0]), beta=1.0, w0=0.0,
                                                  kind=0))
    info = _check_assembly(gp, ctx, w)
    assert info["nnz"] < 9 * len(X)


def test_assembly_degenerate_inputs(gp, ctx):
    rng = np.random.default_rng(5)
    hyper = dict(d=3, r=0.3, sigma2=1e-2, centers=np.array([[0.5, 0.5, 0.5]]), radii=np.array([2.0]),
                 amps=np.array([1.0]), beta=1.0, w0=0.0, kind=0)
    # one point, two points
    for n in (1, 2):
        X = rng.random((n, 3))
        _check_assembly(gp, ctx, dict(X=X, hyper=hyper))
    # duplicates and everything inside one cell
    X = rng.random((300, 3)) * 0.05
    X[100:150] = X[0]
    _check_assembly(gp, ctx, dict(X=X, hyper=hyper))
    # points on cell boundaries (coordinates multiples of r)
    X = np.floor(rng.random((2000, 3)) * 10) * 0.3
    X = X + rng.integers(0, 2, (2000, 3)) * 1e-17
    _check_assembly(gp, ctx, dict(X=X, hyper=hyper))


def test_assembly_clusters_3d_full_size_sampled_rows(gp, ctx):
    """1M-point clustered workload (the benchmark's configuration): GPU rows vs oracle brute force
    on sampled rows; pattern bit-exact, values within tolerance."""
    import oracle
    w = W.clusters_3d(0)
    h = gp.Hyper(**w["hyper"])
    X = torch.tensor(w["X"], dtype=torch.float64, device="cuda")
    info = ctx.assemble(X, h, gp.default_opts())
    assert 85 < info["nnz"] / info["n"] < 115
    c = ctx.csr()
    rp = c["rowptr"].cpu().numpy().astype(np.int64)
    col = c["col"].cpu().numpy().astype(np.int64)
    perm = c["perm"].cpu().numpy().astype(np.int64)
    s = c["dscale"].cpu().numpy()
    v32 = c["val32"].cpu().numpy().astype(np.float64)
    v64 = c["val64"].cpu().numpy()
    iperm = np.empty_like(perm)
    iperm[perm] = np.arange(len(perm))
    rng = np.random.default_rng(1)
    rows = rng.choice(len(perm), 96, replace=False)
    ho = oracle.Hyper(**w["hyper"])
    ref = oracle.rows_brute(w["X"], ho, rows)
    for r, (oc, ov) in zip(rows, ref):
        i = iperm[r]
        cs = col[rp[i]:rp[i + 1]]
        oc_g = np.sort(perm[cs])
        assert np.array_equal(oc_g, oc)
        order = np.argsort(perm[cs])
        a64 = v64[rp[i]:rp[i + 1]][order] / (s[i] * s[cs][order])
        a32 = v32[rp[i]:rp[i + 1]][order] / (s[i] * s[cs][order])
        scale = max(np.abs(ov).max(), 1e-300)
        assert np.abs(a64 - ov).max() <= 1e-12 * scale
        assert np.abs(a32 - ov).max() <= 1e-6 * scale


def test_assembly_sphere_4d_full_size_sampled_rows(gp, ctx):
    """10M-point 4-D workload (599 M stored entries, the benchmark's largest configuration): GPU
    rows vs oracle brute force over all 10M points on sampled rows; pattern bit-exact, values
    within tolerance."""
    import oracle
    w = W.sphere_4d(0)
    h = gp.Hyper(**w["hyper"])
    X = torch.tensor(w["X"], dtype=torch.float64, device="cuda")
    info = ctx.assemble(X, h, gp.default_opts())
    assert 55 < info["nnz"] / info["n"] < 65
    c = ctx.csr()
    rng = np.random.default_rng(2)
    rows = rng.choice(info["n"], 24, replace=False)
    perm = c["perm"].cpu().numpy().astype(np.int64)
    iperm = np.empty_like(perm)
    iperm[perm] = np.arange(len(perm))
    sorted_rows = torch.tensor(iperm[rows], device="cuda")
    rp = c["rowptr"]
    ref = oracle.rows_brute(w["X"], oracle.Hyper(**w["hyper"]), rows)
    s = c["dscale"]
    for k, (oc, ov) in enumerate(ref):
        i = int(sorted_rows[k])
        b, e = int(rp[i]), int(rp[i + 1])
        cs = c["col"][b:e].long()
        pc = perm[cs.cpu().numpy()]
        order = np.argsort(pc)
        assert np.array_equal(pc[order], oc)
        den = (s[i] * s[cs]).cpu().numpy()[order]
        a64 = c["val64"][b:e].cpu().numpy()[order] / den
        a32 = c["val32"][b:e].cpu().numpy().astype(np.float64)[order] / den
        scale = max(np.abs(ov).max(), 1e-300)
        assert np.abs(a64 - ov).max() <= 1e-12 * scale
        assert np.abs(a32 - ov).max() <= 1e-6 * scale


def test_solve_clusters_3d_full_size_sampled_residual_rows(gp, ctx):
    """1M-point benchmark configuration, mixed precision with FP64 refinement: the residual
    y - A a on sampled rows, with the rows of A from oracle brute force over all points, stays
    within the 1e-8 relative bound of the whole residual (each |r_i| <= |r|)."""
    import oracle
    w = W.clusters_3d(0)
    h = gp.Hyper(**w["hyper"])
    ctx.assemble(torch.tensor(w["X"], device="cuda"), h, gp.default_opts())
    a, info = ctx.solve(torch.tensor(w["y"], device="cuda"))
    assert info["relres"] <= 1e-8
    a = a.cpu().numpy()
    rows = np.random.default_rng(3).choice(len(a), 64, replace=False)
    ynorm = np.linalg.norm(w["y"])
    for r, (oc, ov) in zip(rows, oracle.rows_brute(w["X"], oracle.Hyper(**w["hyper"]), rows)):
        assert abs(w["y"][r] - float(ov @ a[oc])) <= 1e-8 * ynorm


# ------------------------------------------------------------------------------------------------
# Solve, log-determinant, LML, gradient
# ------------------------------------------------------------------------------------------------
def _oracle_residual(w, a):
    import oracle
    ho = oracle.Hyper(**w["hyper"])
    csr = oracle.assemble(w["X"], ho)
    return np.linalg.norm(w["y"] - csr.matmat(a)) / np.linalg.norm(w["y"])


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_solve_reaches_refined_residual(gp, ctx, precision):
    w = W.random_small(300, 12000, 3, L=3, sigma2=1e-3, clustered=True)
    h = gp.Hyper(**w["hyper"])
    opts = gp.default_opts(precision=gp.PREC_MIXED if precision == "mixed" else gp.PREC_FP64)
    ctx.assemble(torch.tensor(w["X"], device="cuda"), h, opts)
    a, info = ctx.solve(torch.tensor(w["y"], device="cuda"))
    a = a.cpu().numpy()
    assert info["relres"] <= 1e-8
    assert _oracle_residual(w, a) <= 1e-8


def test_lml_exact_small_2d_matches_oracle(gp, ctx):
    import oracle
    w = W.small_2d(0)
    h = gp.Hyper(**w["hyper"])
    opts = gp.default_opts(precision=gp.PREC_FP64, logdet=gp.LOGDET_EXACT)
    lml, info = ctx.lml(w["X"], w["y"], h, opts)
    e = oracle.lml_exact(w["X"], w["y"], oracle.Hyper(**w["hyper"]))
    assert info["logdet"] == pytest.approx(e["logdet"], rel=1e-10)
    assert info["quad"] == pytest.approx(e["quad"], rel=1e-8)
    assert lml == pytest.approx(e["lml"], rel=1e-8)
    assert info["relres"] <= 1e-8


@pytest.mark.parametrize("precond", [1, 2])
def test_logdet_slq_matches_oracle_with_identical_probes(gp, ctx, precond):
    import oracle
    w = W.random_small(301, 6000, 2, L=3, sigma2=1e-3)
    h = gp.Hyper(**w["hyper"])
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=32, lanczos_steps=60, seed=11, precond=precond)
    lml, info = ctx.lml(w["X"], w["y"], h, opts)
    s = oracle.lml_slq(w["X"], w["y"], oracle.Hyper(**w["hyper"]), m=32, k=60, seed=11, grad=False)
    assert info["logdet"] == pytest.approx(s["logdet"], rel=1e-3)
    assert info["quad"] == pytest.approx(s["quad"], rel=1e-7)
    assert lml == pytest.approx(s["lml"], rel=1e-3)
    # and the estimate is within a few standard errors of the exact value
    e = oracle.lml_exact(w["X"], w["y"], oracle.Hyper(**w["hyper"]))
    assert abs(info["logdet"] - e["logdet"]) <= 5 * info["logdet_stderr"] + 1e-9 * abs(e["logdet"])


@pytest.mark.parametrize("n,d,r", [(1, 1, 0.1), (2, 2, 2.0), (31, 1, 0.05), (32, 2, 2.0), (33, 3, 0.3), (64, 1, 0.02), (65, 2, 0.1),
                                   (97, 3, 2.0), (513, 1, 0.004), (1000, 1, 0.03), (1025, 2, 0.05), (2111, 3, 0.12)])
def test_tiled_cholesky_at_tile_edges(gp, ctx, n, d, r):
    """The exact log-determinant and solve by 32-row tiles: one row, sizes around a tile and several
    tiles, a diagonal-like and a banded matrix, a full one (r = 2), tile fill in 2-D and 3-D.  FP64 on both
    sides: n^2 products of rounding 1.1e-16, a condition number of at most a few 1e3 on the log scale."""
    import oracle
    w = W.random_small(700 + n, n, d, L=3, sigma2=1e-2, r=r)
    opts = gp.default_opts(precision=gp.PREC_FP64, logdet=gp.LOGDET_EXACT)
    lml, info = ctx.lml(w["X"], w["y"], gp.Hyper(**w["hyper"]), opts)
    e = oracle.lml_exact(w["X"], w["y"], oracle.Hyper(**w["hyper"]))
    assert info["logdet"] == pytest.approx(e["logdet"], rel=1e-10, abs=1e-10 * n)
    assert info["quad"] == pytest.approx(e["quad"], rel=1e-10)
    assert lml == pytest.approx(e["lml"], rel=1e-10, abs=1e-9)
    assert info["relres"] <= 1e-12      # the residual is formed from this call's right-hand side and solution


@pytest.mark.parametrize("n,d,row,r", [(12_000, 2, 60, None), (9_001, 3, 60, None), (4_097, 2, 0, 3.0)])
def test_tiled_cholesky_with_much_fill(gp, ctx, n, d, row, r):
    """Larger tile graphs than the ones above (2-D, 3-D with its heavy fill, every tile present): long lists of
    products per tile, more tasks than resident CTAs.  The reference is the dense Cholesky factor of the same
    matrix in FP64; n rounding errors of 1.1e-16 on each of n pivots' logarithms stay below 1e-11 n."""
    w = W.random_small(720 + n, n, d, L=3, sigma2=1e-2, r=r)
    if r is None:
        w["hyper"]["r"] *= (row / 30.0) ** (1.0 / d)
    opts = gp.default_opts(precision=gp.PREC_FP64, logdet=gp.LOGDET_EXACT)
    _, info = ctx.lml(w["X"], w["y"], gp.Hyper(**w["hyper"]), opts)
    assert info["relres"] <= 1e-12
    c = ctx.csr()
    A = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    rows = torch.repeat_interleave(torch.arange(n, device="cuda"), c["rowptr"].diff())
    A[rows, c["col"].long()] = c["val64"]
    ref = 2.0 * torch.linalg.cholesky(A).diagonal().log().sum().item()
    assert ctx.logdet()[2]["logdet_hat"] == pytest.approx(ref, abs=1e-11 * n)


@pytest.mark.parametrize("steps,rel", [(1, 1e-9), (2, 1e-9), (33, 1e-9), (257, 1e-6), (300, 1e-6)])
def test_slq_quadrature_matches_the_oracle_eigensolve(gp, ctx, steps, rel):
    """The quadrature of log T without its eigen-decomposition against the oracle's Gauss quadrature, in
    FP64 with identical probes: one and two steps, a few tens, and more rows of T than the CTA has
    threads.  Up to 33 steps T agrees to rounding (1e-13 per entry, times T's condition number of
    at most 1e4); beyond that the two Lanczos processes lose orthogonality at different steps."""
    import oracle
    w = W.random_small(303, 3000, 2, L=3, sigma2=1e-2)
    opts = gp.default_opts(precision=gp.PREC_FP64, logdet=gp.LOGDET_SLQ, probes=16, lanczos_steps=steps, seed=4)
    _, info = ctx.lml(w["X"], w["y"], gp.Hyper(**w["hyper"]), opts)
    s = oracle.lml_slq(w["X"], w["y"], oracle.Hyper(**w["hyper"]), m=16, k=steps, seed=4, grad=False)
    assert info["logdet"] == pytest.approx(s["logdet"], rel=rel)


@pytest.mark.parametrize("precond", [1, 2])
def test_gradient_matches_oracle_hutchinson(gp, ctx, precond):
    import oracle
    w = W.random_small(302, 4000, 2, L=3, sigma2=1e-3)
    h = gp.Hyper(**w["hyper"])
    opts = gp.default_opts(probes=32, lanczos_steps=50, seed=5, tol_probe=1e-6, precond=precond)
    lml, g, info = ctx.lml_grad(w["X"], w["y"], h, opts)
    s = oracle.lml_slq(w["X"], w["y"], oracle.Hyper(**w["hyper"]), m=32, k=50, seed=5)
    gref = s["grad"]
    # measured on GB300: 2.5e-9 of max |g| for both preconditioners (FP32 probe solves to 1e-6,
    # FP64 refinement of a); the bar keeps a wide margin for other GPUs and drivers
    assert np.abs(g - gref).max() <= 1e-6 * np.abs(gref).max()


def test_gradient_fp64_form_matches_oracle_hutchinson_tightly(gp, ctx):
    """The adjoint contraction itself, without FP32 solves in the way: the plain FP64 form with
    y and probe solves to 1e-11 against the oracle's FP64 Hutchinson gradient (identical probes,
    its CG to 1e-12) agrees to 1e-6 of the largest component."""
    import oracle
    w = W.random_small(304, 3000, 3, L=3, sigma2=1e-3)
    h = gp.Hyper(**w["hyper"])
    opts = gp.default_opts(precision=gp.PREC_FP64, logdet=gp.LOGDET_SLQ, probes=32, lanczos_steps=50, seed=6,
                           tol_probe=1e-11, tol_refine=1e-11, precond=1)
    lml, g, info = ctx.lml_grad(w["X"], w["y"], h, opts)
    s = oracle.lml_slq(w["X"], w["y"], oracle.Hyper(**w["hyper"]), m=32, k=50, seed=6, tol=1e-12)
    gref = s["grad"]
    assert g.shape == gref.shape == (h.nparams,)
    assert np.abs(g - gref).max() <= 1e-6 * np.abs(gref).max()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_slq_when_the_krylov_space_is_exhausted(gp, ctx, precision):
    """Degenerate SLQ cases: n = 40 points (fewer than the 100 Lanczos steps) and isolated points
    (A diagonal, Ah = I).  The probe columns stop when their residual reaches the rounding level
    instead of reporting a breakdown; the log-determinant matches the oracle with identical probes,
    and for the diagonal case equals sum log A_ii exactly."""
    import oracle
    prec = gp.PREC_MIXED if precision == "mixed" else gp.PREC_FP64
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=32, lanczos_steps=100, seed=3, precision=prec)
    w = W.random_small(440, 40, 2, L=2, sigma2=1e-2)
    lml, g, info = ctx.lml_grad(w["X"], w["y"], gp.Hyper(**w["hyper"]), opts)
    s = oracle.lml_slq(w["X"], w["y"], oracle.Hyper(**w["hyper"]), m=32, k=100, seed=3)
    assert info["logdet"] == pytest.approx(s["logdet"], rel=1e-3)
    assert np.abs(g - s["grad"]).max() <= 1e-6 * np.abs(s["grad"]).max()
    rng = np.random.default_rng(7)
    X = rng.random((500, 2))
    y = np.sin(6 * X[:, 0])
    hyper = dict(d=2, r=1e-6, sigma2=1e-2, centers=np.array([[0.5, 0.5]]), radii=np.array([2.0]),
                 amps=np.array([1.0]), beta=1.0, w0=0.0, kind=0)
    lml, g, info = ctx.lml_grad(X, y, gp.Hyper(**hyper), opts)
    e = oracle.lml_exact(X, y, oracle.Hyper(**hyper))
    assert info["nnz"] == 500
    assert info["logdet"] == pytest.approx(e["logdet"], rel=1e-12)
    assert lml == pytest.approx(e["lml"], rel=1e-10)


def test_graph_replay_equals_eager_launches(gp, monkeypatch):
    """Runs of CG iterations replayed as CUDA graphs give bit-identical results to launching every
    kernel eagerly (the same kernels with the same arguments), and count the same launches."""
    w = W.random_small(305, 6000, 3, L=3, sigma2=1e-3)
    h = gp.Hyper(**w["hyper"])
    X = torch.tensor(w["X"], device="cuda")
    y = torch.tensor(w["y"], device="cuda")
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=64, lanczos_steps=50, seed=8)
    monkeypatch.setenv("GP2S_GRAPHS", "1")
    lml_g, g_g, info_g = gp.Context(0).lml_grad(X, y, h, opts)
    monkeypatch.setenv("GP2S_GRAPHS", "0")
    lml_e, g_e, info_e = gp.Context(0).lml_grad(X, y, h, opts)
    assert lml_g == lml_e
    assert np.array_equal(g_g, g_e)
    assert info_g["iters_y"] == info_e["iters_y"] and info_g["launches"] == info_e["launches"]


@pytest.mark.parametrize("probes,n", [(16, 40_003), (32, 160_003), (64, 40_003)])
def test_spmm_gather_copies_equal_register_gathers(gp, monkeypatch, probes, n):
    """The RB8 SpMM's forms (the gathered probe rows all loaded into registers; or 16 or all 32 of
    every batch's rows brought into shared memory by tensor-map gather copies) run the same FMAs in
    the same order and reduce every tile's dots in tile order: a whole mixed-precision evaluation
    of clustered 3-D points (thousands of 8-row blocks, a ragged last block; at 160,003 points the
    multi-segment dot reduction) gives the same LML, gradient and iteration counts bit for bit."""
    w = W.clusters_3d(3, n=n)
    h = gp.Hyper(**w["hyper"])
    X = torch.tensor(w["X"], device="cuda")
    y = torch.tensor(w["y"], device="cuda")
    opts = gp.default_opts(probes=probes, lanczos_steps=30, seed=5)
    out = []
    for tma in ("0", "16", "32"):
        monkeypatch.setenv("GP2S_SPMM_TMA", tma)
        out.append(gp.Context(0).lml_grad(X, y, h, opts))
    l0, g0, i0 = out[0]
    for l1, g1, i1 in out[1:]:
        assert l1 == l0 and np.array_equal(g1, g0)
        assert (i1["iters_y"], i1["iters_probes"]) == (i0["iters_y"], i0["iters_probes"])
    if n > 100_000:
        assert i0["spmm_seg_tiles"] > 1


@pytest.mark.parametrize("probes,n,row", [(16, 33, 12), (16, 3001, 33), (16, 2500, 120), (48, 1500, 31)])
def test_fp64_spmm_with_partly_filled_warps(gp, ctx, probes, n, row):
    """FP64 multi-RHS SpMM where the columns do not fill a warp (16: the half-warps take alternate entries of a
    row; 48: 24 lanes): rows of odd lengths, beyond one 32-entry batch, a matrix smaller than the grid.
    Probe solves to 1e-10 on both sides leave about 1e-8 of the gradient."""
    import oracle
    w = W.random_small(760 + n, n, 2, L=3, sigma2=1e-2)
    w["hyper"]["r"] *= (row / 30.0) ** 0.5
    opts = gp.default_opts(precision=gp.PREC_FP64, logdet=gp.LOGDET_SLQ, probes=probes, lanczos_steps=20, seed=6,
                           tol_probe=1e-10)
    lml, g, info = ctx.lml_grad(w["X"], w["y"], gp.Hyper(**w["hyper"]), opts)
    s = oracle.lml_slq(w["X"], w["y"], oracle.Hyper(**w["hyper"]), m=probes, k=20, seed=6, tol=1e-12)
    assert info["logdet"] == pytest.approx(s["logdet"], rel=1e-8)
    assert np.abs(g - s["grad"]).max() <= 1e-7 * np.abs(s["grad"]).max()


@pytest.mark.parametrize("n,row", [(1, 1), (33, 5), (2049, 150), (20_000, 40), (60_001, 180)])
def test_band_matrix_y_solve(gp, ctx, n, row):
    """One-dimensional points in SLQ evaluations without a gradient: y by the tiled Cholesky factor of the
    band, with the residual of an FP64 solve, and the same evaluation through y's PCG (lml_grad, whose y
    solve meets 1e-8: its quadratic term agrees to second order in that).  A point, a band as wide as the
    matrix, rows of several tiles."""
    w = W.random_small(780 + n, n, 1, L=3, sigma2=1e-3, r=0.05 if n == 1 else None)
    w["hyper"]["r"] *= row / 30.0
    h = gp.Hyper(**w["hyper"])
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=16, lanczos_steps=min(40, max(1, n // 2)), seed=3)
    lml, info = ctx.lml(w["X"], w["y"], h, opts)
    assert info["iters_y"] == 0 and info["relres"] <= 1e-10
    lml_g, _, info_g = ctx.lml_grad(w["X"], w["y"], h, opts)
    assert info["quad"] == pytest.approx(info_g["quad"], rel=1e-7)
    assert info["logdet"] == pytest.approx(info_g["logdet"], rel=1e-6, abs=1e-6)
    assert ctx.logdet()[0] == pytest.approx(info["logdet"], rel=1e-9, abs=1e-9)


@pytest.mark.parametrize("bj", [64, 128])
@pytest.mark.parametrize("n", [1, 2, 8, 9, 31, 33, 63, 64, 65, 100, 127, 128, 129, 200, 1031])
def test_block_jacobi_factors_at_block_edges(gp, ctx, bj, n):
    """A matrix of one block (partly filled panels, rows past n): M is A, so a step leaves the error of
    M^{-1} in FP32, at most n eps kappa = 128 * 6e-8 * 1000 < 1e-2, and four steps reach the first tolerance
    (1e-6) and each restart's.  More blocks, the last one ragged: the FP64 residual, formed here from the
    CSR."""
    w = W.random_small(830 + n, n, 2, L=3, sigma2=0.1, r=0.6 if n < 8 else None)
    h = gp.Hyper(**w["hyper"])
    ctx.assemble(w["X"], h, gp.default_opts(precond=2, bj_block=bj))
    key, A64, _, _, _ = _csr_orig(ctx.csr())
    A = np.zeros(n * n)
    A[key] = A64
    a, info = ctx.solve(w["y"])
    assert info["relres"] <= 1e-8
    assert np.linalg.norm(w["y"] - A.reshape(n, n) @ a) <= 2e-8 * np.linalg.norm(w["y"])
    if n <= bj:
        assert info["iters"] <= 4 * (info["outer"] + 1)


@pytest.mark.parametrize("bj", [64, 128])
@pytest.mark.parametrize("blocks,rest", [(2, 0), (2, 1), (3, 37), (8, 63), (160, 5)])
def test_block_jacobi_factors_of_every_block(gp, ctx, bj, blocks, rest):
    """Points in one dimension in clusters of a block's rows, further apart than the support: M is A again, block
    by block, the last one ragged, and the few-step bound of a single block holds for all of them.  A block
    that is wrong, or taken from other rows, needs more."""
    n, r = bj * blocks + rest, 1e-3
    w = W.random_small(840 + n, n, 1, L=3, sigma2=0.1, r=r)
    rng = np.random.default_rng(n)
    w["X"][:, 0] = (np.arange(n) // bj) * 4 * r + 0.8 * r * rng.random(n)
    order = rng.permutation(n)
    h = gp.Hyper(**w["hyper"])
    info = ctx.assemble(w["X"][order], h, gp.default_opts(precond=2, bj_block=bj))
    assert info["nnz"] == bj * bj * blocks + rest * rest
    _, s = ctx.solve(w["y"][order])
    assert s["relres"] <= 1e-8
    assert s["iters"] <= 4 * (s["outer"] + 1)


def test_autograd_function(gp, ctx):
    w = W.random_small(303, 3000, 2, L=2, sigma2=1e-3)
    h = gp.Hyper(**w["hyper"])
    theta = torch.tensor(h.theta(), dtype=torch.float64, requires_grad=True)
    X = torch.tensor(w["X"], device="cuda")
    y = torch.tensor(w["y"], device="cuda")
    opts = gp.default_opts(probes=32, seed=2)
    out = gp.GP2SLML.apply(theta, X, y, h, opts)
    out.backward()
    lml, g, _ = ctx.lml_grad(X, y, h, opts)
    assert float(out) == pytest.approx(lml, rel=1e-12)
    np.testing.assert_allclose(theta.grad.numpy(), g, rtol=1e-12)


def test_invalid_arguments_are_reported(gp, ctx):
    w = W.random_small(304, 100, 2)
    h = gp.Hyper(**w["hyper"])
    bad = gp.Hyper(**{**w["hyper"], "r": -1.0})
    with pytest.raises(gp.GP2SError) as e:
        ctx.assemble(w["X"], bad)
    assert e.value.status == gp.EINVAL
    X = w["X"].copy()
    X[3, 1] = np.nan
    with pytest.raises(gp.GP2SError) as e:
        ctx.assemble(X, h)
    assert e.value.status == gp.EINVAL
    with pytest.raises(gp.GP2SError) as e:
        ctx.lml(w["X"], w["y"], h, gp.default_opts(probes=33))
    assert e.value.status == gp.EINVAL
    # a zero diagonal (sigma2 = 0, point outside every bump, w0 = 0) is not positive definite
    far = gp.Hyper(**{**w["hyper"], "sigma2": 0.0, "centers": np.full((3, 2), 50.0)})
    with pytest.raises(gp.GP2SError) as e:
        ctx.assemble(w["X"], far)
    assert e.value.status == gp.ENOTPD


# ------------------------------------------------------------------------------------------------
# Block-Jacobi preconditioned path (opts.precond = 2, the default in MIXED precision)
# ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("bj", [0, 128])
def test_block_jacobi_solve_logdet_and_gradient(gp, ctx, bj):
    """Properties that hold for any preconditioner: the y solve reaches the FP64 residual against
    the oracle's A; the preconditioned SLQ log-determinant agrees with the exact one within its
    standard error; the Hutchinson gradient agrees with the exact gradient within its noise."""
    import oracle
    w = W.random_small(310, 3000, 2, L=3, sigma2=1e-3, r=0.05)
    h = gp.Hyper(**w["hyper"])
    X = torch.tensor(w["X"], device="cuda")
    y = torch.tensor(w["y"], device="cuda")
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=128, lanczos_steps=100, seed=3, precond=2, bj_block=bj)
    lml, g, info = ctx.lml_grad(X, y, h, opts)
    ho = oracle.Hyper(**w["hyper"])
    e = oracle.lml_exact(w["X"], w["y"], ho)
    assert info["relres"] <= 1e-8
    assert info["quad"] == pytest.approx(e["quad"], rel=1e-7)
    assert abs(info["logdet"] - e["logdet"]) <= 5 * info["logdet_stderr"] + 1e-9 * abs(e["logdet"])
    gex = oracle.grad_exact(w["X"], w["y"], ho)
    # the a^T dA a part is exact; the trace part is a 128-probe estimate
    err = np.abs(g - gex)
    assert np.median(err / (np.abs(gex) + 1e-3 * np.abs(gex).max())) < 0.1
    # fewer iterations than plain Jacobi on the same problem
    _, _, info1 = ctx.lml_grad(X, y, h, gp.default_opts(logdet=gp.LOGDET_SLQ, probes=128, lanczos_steps=100,
                                                         seed=3, precond=1))
    assert info["iters_probes"] < info1["iters_probes"]
