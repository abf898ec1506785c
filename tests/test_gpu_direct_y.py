"""The y solve of one-dimensional points by the tiled Cholesky factor (SLQ evaluations without a gradient):
what choosing it costs, and what happens where it cannot or should not run."""
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


def _line(n, row, sigma2):
    """n points in one dimension on the GPU with about `row` stored entries per row."""
    w = W.random_small(910 + n, n, 1, L=3, sigma2=sigma2)
    w["hyper"]["r"] *= row / 30.0
    return torch.tensor(w["X"], device="cuda"), torch.tensor(w["y"], device="cuda"), w["hyper"]


def test_a_new_pattern_is_ordered_in_little_time(gp):
    """A step that moves r has a new pattern, whose elimination order is found on the host while the GPU
    waits.  On a band of 5,625 tile rows that is a few ms of an evaluation of about 14; going through all tiles
    at every step made the evaluation five times as long as one on the same pattern."""
    X, y, hyper = _line(180_000, 40, 1e-3)
    ctx = gp.Context(0)
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=16, lanczos_steps=100, seed=3)
    r = hyper["r"]

    def solve_ms(step):
        h = gp.Hyper(**dict(hyper, r=r * (1.0 + 1e-4 * step)))
        info = ctx.lml(X, y, h, opts)[1]
        assert info["iters_y"] == 0 and info["relres"] <= 1e-10
        return info["ms_solve"]

    solve_ms(0)
    new = min(solve_ms(step) for step in range(1, 5))
    same = min(solve_ms(4) for _ in range(4))
    assert new < 2.0 * same


def test_a_matrix_that_the_factorisation_refuses_keeps_y_beside_the_probes(gp, monkeypatch):
    """Past the size that the exact factorisation takes (8 n^2 bytes against GP2S_MEM_LIMIT) the y column shares
    the probes' steps from the first one.  An evaluation with the gradient, which never factors, does the same
    solves when its probes need not converge: the same steps, bit for bit (y's steps on their own go through
    another matrix kernel, whose sums run in another order)."""
    X, y, hyper = _line(20_000, 40, 1e-3)
    h = gp.Hyper(**hyper)
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=16, lanczos_steps=100, seed=3, tol_probe=1.0)
    free = gp.Context(0).lml(X, y, h, opts)[1]
    monkeypatch.setenv("GP2S_MEM_LIMIT", str(1 << 30))
    ctx = gp.Context(0)
    info = ctx.lml(X, y, h, opts)[1]
    with_grad = ctx.lml_grad(X, y, h, opts)[2]
    assert info["iters_y"] == with_grad["iters_y"] > 0 and info["relres"] == with_grad["relres"] <= 1e-8
    assert info["quad"] == with_grad["quad"]
    assert info["iters_probes"] == free["iters_probes"] and info["logdet"] == pytest.approx(free["logdet"], rel=1e-12)
    assert info["quad"] == pytest.approx(free["quad"], rel=1e-7)


@pytest.mark.parametrize("n,row,sigma2", [(30_000, 300, 100.0), (100_000, 100, 100.0), (65_536, 200, 10.0)])
def test_a_system_of_few_iterations_is_not_factored(gp, n, row, sigma2):
    """A large noise variance leaves PCG a handful of iterations, beside the probes' steps, where the factor of
    these bands takes 4 to 7 ms.  The evaluation with the gradient, which never factors, takes the same steps."""
    X, y, hyper = _line(n, row, sigma2)
    h = gp.Hyper(**hyper)
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=16, lanczos_steps=100, seed=3, tol_probe=1.0)
    ctx = gp.Context(0)
    info = ctx.lml(X, y, h, opts)[1]
    with_grad = ctx.lml_grad(X, y, h, opts)[2]
    assert 0 < info["iters_y"] <= 60 and info["iters_y"] == with_grad["iters_y"]
    assert info["quad"] == with_grad["quad"] and info["relres"] == with_grad["relres"] <= 1e-8
    assert info["logdet"] == with_grad["logdet"] and info["iters_probes"] == with_grad["iters_probes"]


@pytest.mark.parametrize("n,row,probes,steps", [(20_000, 40, 16, 100), (20_000, 40, 48, 7), (65_000, 200, 64, 20), (9000, 300, 32, 8)])
def test_a_y_column_given_up_leaves_the_probes_as_they_are(gp, n, row, probes, steps):
    """y starts beside the probes, does not converge and is left to the factor: at the check after eight
    steps, with the probes at their end or on their way.  Their records are those of the log-determinant
    alone, whose y column is idle from the first step."""
    X, y, hyper = _line(n, row, 1e-3)
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=probes, lanczos_steps=steps, seed=3)
    ctx = gp.Context(0)
    info = ctx.lml(X, y, gp.Hyper(**hyper), opts)[1]
    assert info["iters_y"] == 0 and info["relres"] <= 1e-10
    assert ctx.logdet()[0] == pytest.approx(info["logdet"], rel=1e-13)


def _least_limit(gp, monkeypatch, call):
    """The least GP2S_MEM_LIMIT, to 1 KB, under which `call` succeeds on a context of its own."""
    lo, hi = 0, 1 << 17
    while hi - lo > 1:
        mid = (lo + hi) // 2
        monkeypatch.setenv("GP2S_MEM_LIMIT", str(mid << 10))
        try:
            call(gp.Context(0))
            hi = mid
        except gp.GP2SError as e:
            assert e.status == gp.ENOMEM
            lo = mid
    monkeypatch.setenv("GP2S_MEM_LIMIT", str(hi << 10))
    return hi << 10


@pytest.mark.parametrize("n,row,steps", [(300, 30, 20), (500, 60, 3), (501, 200, 100)])
def test_a_factor_without_room_leaves_y_to_pcg(gp, monkeypatch, n, row, steps):
    """Under the least limit that the evaluation itself fits in, the factor's buffers are refused after the
    probes have run: y's PCG follows on its own, with the same probe records and the same results."""
    X, y, hyper = _line(n, row, 1e-3)
    h = gp.Hyper(**hyper)
    opts = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=16, lanczos_steps=steps, seed=3)
    free = gp.Context(0).lml(X, y, h, opts)[1]
    assert free["iters_y"] == 0
    limit = _least_limit(gp, monkeypatch, lambda c: c.lml(X, y, h, opts))
    assert limit >= 8 * n * n          # the factorisation is tried
    ctx = gp.Context(0)
    for _ in range(2):
        info = ctx.lml(X, y, h, opts)[1]
        assert info["iters_y"] > 0 and info["relres"] <= 1e-8
        assert info["iters_probes"] == free["iters_probes"]
        assert info["logdet"] == pytest.approx(free["logdet"], rel=1e-13)
        assert info["quad"] == pytest.approx(free["quad"], rel=1e-7)


@pytest.mark.parametrize("n", [300, 500])
def test_a_factor_under_a_limit_takes_no_room_from_later_calls(gp, monkeypatch, n):
    """A larger call (four times the probes, with the gradient) that fits the limit on a fresh context still
    fits after an evaluation whose y solve took the factor."""
    X, y, hyper = _line(n, 30, 1e-3)
    h = gp.Hyper(**hyper)
    small = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=16, lanczos_steps=20, seed=3)
    large = gp.default_opts(logdet=gp.LOGDET_SLQ, probes=64, lanczos_steps=20, seed=3)
    _least_limit(gp, monkeypatch, lambda c: c.lml_grad(X, y, h, large))
    ctx = gp.Context(0)
    assert ctx.lml(X, y, h, small)[1]["iters_y"] == 0
    ctx.lml_grad(X, y, h, large)
