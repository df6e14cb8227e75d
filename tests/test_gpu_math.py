"""The float64 functions of the kernels that stand in for the library's (csrc/rpb_internal.cuh, csrc/pair_math.cuh), compiled
by themselves, against long double (128 bits on the GPU's host)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1612_00474_gb300", "csrc")
FUNCTIONS = ("rsqrt_pos", "rcp_pos", "root", "inverse", "exp_table", "exp_neg")
SRC = r"""
#include "pair_math.cuh"
using namespace rpb;
__global__ void evaluate(int which, const double *x, double *y, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double root, inverse;
    root_and_inverse(x[i], &root, &inverse);
    if (which >= 4)
        y[i] = which == 4 ? exp_table(x[i]) : exp_neg(x[i]);
    else
        y[i] = which == 0 ? rsqrt_pos(x[i]) : which == 1 ? rcp_pos(x[i]) : which == 2 ? root : inverse;
}
extern "C" int run(int which, const void *x, void *y, int n)
{
    evaluate<<<(n + 255) / 256, 256>>>(which, (const double *)x, (double *)y, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    from paper_1612_00474_gb300 import build

    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("long double is no wider than float64")
    d = tmp_path_factory.mktemp("math")
    (d / "m.cu").write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    str(d / "m.cu"), "-o", str(d / "m.so")], check=True)
    lib = ctypes.CDLL(str(d / "m.so"))

    def call(name, x):
        a = torch.tensor(x, dtype=torch.float64, device="cuda")
        b = torch.empty_like(a)
        assert lib.run(FUNCTIONS.index(name), ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(b.data_ptr()), len(x)) == 0
        return b.cpu().numpy()

    return call


def _positive(lo, hi):
    """Mantissas all over, at both ends of a power of two and its neighbours, exponents lo .. hi."""
    rng = np.random.default_rng(7)
    m = np.concatenate([1.0 + rng.random(200000), 1.0 + 2.0 ** -rng.integers(1, 53, 2000), 2.0 - 2.0 ** -rng.integers(1, 53, 2000)])
    e = np.concatenate([rng.integers(-3, 4, 100000), rng.integers(lo, hi + 1, len(m) - 100000)])
    return np.ldexp(np.minimum(m, np.nextafter(2.0, 1.0)), e)


def _ulps(y, exact):
    return np.abs((y.astype(np.longdouble) - exact) / np.spacing(np.abs(exact).astype(np.float64)).astype(np.longdouble))


# one rounding of the result, 0.5, and what the step of the approximation leaves: 2^-58.7 of a root and 2^-59.7 of a
# reciprocal, 0.02 and 0.01 at most, with 0.01 for the roundings inside the correction
@pytest.mark.parametrize("name,of,bound", [("rsqrt_pos", lambda x: 1 / np.sqrt(x), 0.53), ("rcp_pos", lambda x: 1 / x, 0.52),
                                           ("root", np.sqrt, 0.51), ("inverse", lambda x: 1 / np.sqrt(x), 0.53)])
def test_roots_and_reciprocals(evaluate, name, of, bound):
    x = _positive(-1021, 998)  # plain_pos: 2^-1022 .. 2^1000 (a reciprocal's result is normal up to 2^1021)
    y = evaluate(name, x)
    assert float(_ulps(y, of(x.astype(np.longdouble))).max()) <= bound


# one rounding, 0.5; the series' next term, (ln 2 / 128)^6 / 720, 0.32 where the result's last place counts least; 0.01 for
# the roundings before the last
def test_exponential(evaluate):
    rng = np.random.default_rng(8)
    n = np.arange(0, 64639)  # every table entry and exponent: in the middle, and where the nearest entry changes
    x = -np.concatenate([n * np.log(2.0) / 64, (n + 0.5) * np.log(2.0) / 64 - 1e-9, (n + 0.5) * np.log(2.0) / 64 + 1e-9,
                         rng.random(200000) * 40, rng.random(200000) * 700, rng.random(20000) * 1e-3,
                         2.0 ** -rng.integers(1, 1000, 2000), [0.0, 700.0]])
    x = x[x >= -700.0]
    exact = np.exp(x.astype(np.longdouble))
    y = evaluate("exp_table", x)
    assert float(_ulps(y, exact).max()) <= 0.83
    inside = (x > -700.0) & (x < 0.0)
    assert np.array_equal(evaluate("exp_neg", x)[inside], y[inside])
    far = np.array([0.0, 1.0, -700.0, -720.0, -745.0, -1e4, -np.inf, np.inf, np.nan])  # the library's
    z = evaluate("exp_neg", far)
    assert np.array_equal(z[[0, 5, 6, 7]], [1.0, 0.0, 0.0, np.inf]) and np.isnan(z[8])
    assert np.allclose(z[1:5], np.exp(far[1:5]), rtol=1e-15, atol=5e-324)
