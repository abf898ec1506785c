"""The library's own FP64 square root and reciprocal (gp2s_kernel_math.cuh) against numpy's correctly rounded
ones, value by value, through a small library compiled here around the header."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "gp2s_kernel_math.cuh"
__global__ void k_apply(int which, const double *in, double *out, long n)
{
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        out[i] = which ? gp2s::rcp_pos(in[i]) : gp2s::sqrt_pos(in[i]);
}
extern "C" int apply(int which, const double *in, double *out, long n)
{
    k_apply<<<256, 256>>>(which, in, out, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def apply(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2512_06143_gb300 import build
    d = tmp_path_factory.mktemp("scalar_math")
    (d / "apply.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", os.path.join(build.HERE, "csrc"), "-shared",
                    str(d / "apply.cu"), "-o", str(d / "libapply.so")], check=True)
    lib = ctypes.CDLL(str(d / "libapply.so"))
    lib.apply.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_long]

    def run(which, values):
        x = torch.from_numpy(np.ascontiguousarray(values)).cuda()
        out = torch.empty_like(x)
        assert lib.apply(which, x.data_ptr(), out.data_ptr(), x.numel()) == 0
        return out.cpu().numpy()

    return run


def _ulps(a, b):
    """Distance of positive doubles in units of the last place."""
    return np.abs(a.view(np.int64) - b.view(np.int64))


def _draw(n, seed):
    rng = np.random.default_rng(seed)
    return np.ldexp(1.0 + rng.random(n), rng.integers(-104, 104, n))


def _edges():
    """Powers of two with their neighbours, over all exponents and so over both ends of the range that the
    quick form takes; the ends of the mantissa's upper 23 bits; zero, subnormals, the largest double."""
    p = np.ldexp(1.0, np.arange(-1022, 1024))
    e = np.concatenate([p, np.nextafter(p, 0.0), np.nextafter(p, np.inf)])
    step = np.ldexp(1.0 + np.arange(0, 1 << 23, 4099) * 2.0 ** -23, 3)
    return np.concatenate([e, step, np.nextafter(step, 0.0), [np.finfo(np.float64).max]])


def test_square_root(apply):
    """Off by less than 2^-80 before its last rounding: of drawn values one in 2^26 may differ from the rounded
    root, by one unit; a root that is a double itself is met."""
    q = _draw(1 << 22, 1)
    d = _ulps(apply(0, q), np.sqrt(q))
    assert d.max() <= 1 and np.count_nonzero(d) <= 4
    rng = np.random.default_rng(2)
    root = rng.integers(1, 1 << 26, 1 << 20).astype(np.float64)
    exact = np.ldexp(root, rng.integers(-30, 20, root.size))
    assert np.array_equal(apply(0, exact * exact), exact)
    outside = np.array([0.0, 5e-324, 1e-310, 2.0 ** -101, 2.0 ** 101, 1e300])
    assert np.array_equal(apply(0, outside), np.sqrt(outside))
    e = _edges()
    assert _ulps(apply(0, e), np.sqrt(e)).max() <= 1


def test_square_root_beside_the_middle_of_two_doubles(apply):
    """Squares of the middles between neighbouring doubles, rounded: their roots are the closest to a rounding
    boundary that there are.  One unit at most."""
    rng = np.random.default_rng(3)
    g = rng.integers(1 << 52, 1 << 53, 20_000)
    q = np.array([float((2 * int(v) + 1) ** 2) for v in g])      # (v + 1/2)^2, rounded, times 4
    q = np.concatenate([q, np.nextafter(q, 0.0), np.nextafter(q, np.inf), np.nextafter(np.ldexp(1.0, np.arange(-98, 100)), 0.0)])
    q = np.ldexp(q, -100 * (q > 2.0 ** 99))
    assert _ulps(apply(0, q), np.sqrt(q)).max() <= 1


def test_reciprocal(apply):
    """Off by less than 2^-65 before its last rounding: at most one unit from the rounded quotient, and equal to
    it but for one value in some 2^11 (2^-65 of the value on either side of a middle, against a unit of
    2^-53 to 2^-52)."""
    d = _draw(1 << 22, 4)
    u = _ulps(apply(1, d), 1.0 / d)
    assert u.max() <= 1 and np.count_nonzero(u) <= d.size >> 10
    e = _edges()
    e = e[(e >= 2.0 ** -1021) & (e <= 2.0 ** 1021)]
    assert _ulps(apply(1, e), 1.0 / e).max() <= 1
    p = np.ldexp(1.0, np.arange(-120, 120))
    assert np.array_equal(apply(1, p), 1.0 / p)
    outside = np.array([3.0 * 2.0 ** -110, 7.0 * 2.0 ** 120, 1e-300, 1e300])
    assert np.array_equal(apply(1, outside), 1.0 / outside)
