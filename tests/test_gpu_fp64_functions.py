"""The FP64 functions of the step (logarithm, exponential, reciprocal and quotients, the limited slope, the sign tests) against
extended precision (numpy's long double: 113 bits on the GPU's Arm host), at the edges of the logarithm's 128 intervals, at the
ends of the ranges that the approximations serve, and on subnormal, infinite and NaN operands, which take CUDA's own functions.

Bounds, in units of the result's last place (ulp) unless they say otherwise:
  log64   the sum k ln 2 - log c (0.5), the final sum (0.5), k times the rounding of ln 2 (0.4 at k = 1) and the small term's
          roundings (below 0.2): 1.6;  CUDA's log on subnormal operands: 1
  exp64   the final sum (0.5) and the roundings of a term below 2^-8 of it: 0.52;  CUDA's exp beyond |x| = 600: 1
  rcp64   the last fused operation (0.5) and e^3 < 2^-59: 0.52
  quot64  that and the product: 2.1 2^-53 relative
  div64   the corrected quotient: 0.52
  theta64 two roundings of an exponent below 2 and the exponential: 4e-16 relative"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu

SRC = r"""
#include "hlbm_split.cuh"
using namespace hlbm;
__global__ void eval(int which, const double *a, const double *b, double *out, int n, const KParams kp)
{
    __shared__ Tables64 tab;
    load_tables64(tab);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double x, y;
        switch (which) {
        case 0: out[i] = log64(tab, a[i]); break;
        case 1: out[i] = exp64(tab, a[i]); break;
        case 2: out[i] = rcp64_ok(a[i]) ? rcp64(a[i]) : 1.0 / a[i]; break;
        case 3: out[i] = quot64(a[i], b[i]); break;
        case 4: div64(a[i], a[i], b[i], x, y); out[i] = x == y || (x != x && y != y) ? x : 12345.0; break;
        case 5: out[i] = va_slope64(a[i], b[i]); break;
        case 6: out[i] = (positive64(a[i]) ? 1.0 : 0.0) + (negative64(a[i]) ? 2.0 : 0.0); break;
        case 7: out[i] = theta64(tab, kp, a[i], b[i]); break;
        }
    }
}
extern "C" int run(int which, const double *a, const double *b, double *out, int n, double gm1, double inv_cv)
{
    KParams kp = {};
    kp.gm1 = gm1;
    kp.inv_cv = inv_cv;
    eval<<<304, 256>>>(which, a, b, out, n, kp);
    return cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess;
}
"""
LOG, EXP, RCP, QUOT, DIV, SLOPE, SIGN, THETA = range(8)


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision on this host")
    from paper_2002_03644_gb300 import build
    d = tmp_path_factory.mktemp("fp64")
    src, lib = str(d / "f.cu"), str(d / "f.so")
    open(src, "w").write(SRC)
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", *build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, "-I", build.INCLUDE,
                    "-o", lib, src], check=True)
    run = ctypes.CDLL(lib).run
    run.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_int] + [ctypes.c_double] * 2

    def f(which, a, b=None, gm1=0.0, inv_cv=0.0):
        a = torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
        b = a if b is None else torch.from_numpy(np.array(np.broadcast_to(b, a.shape), dtype=np.float64)).cuda()
        out = torch.empty_like(a)
        torch.cuda.synchronize()
        assert run(which, a.data_ptr(), b.data_ptr(), out.data_ptr(), a.numel(), gm1, inv_cv) == 0
        return out.cpu().numpy()
    return f


def ulps(got, ref):
    return np.abs(got.astype(np.longdouble) - ref) / np.spacing(np.maximum(np.abs(got), np.abs(ref.astype(np.float64))))


def near(x, k=3):
    """x and its k neighbours on each side."""
    x = np.atleast_1d(np.asarray(x, dtype=np.float64))
    bits = x.view(np.int64)
    return np.concatenate([(bits + d).view(np.float64) for d in range(-k, k + 1)])


def spread(rng, n, lo, hi):
    """Random mantissas with exponents lo .. hi - 1."""
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))


RNG = np.random.default_rng(5)
EDGES = near(1.0 + np.arange(128) / 128.0)


@pytest.mark.parametrize("x", [
    EDGES, np.ldexp(EDGES, -1), EDGES * 4.0, np.ldexp(EDGES, 1000), np.ldexp(EDGES, -1000), near(1.0, 60),
    RNG.uniform(0.5, 2.0, 200000), spread(RNG, 100000, -1021, 1023),
], ids=["1..2", "half", "quadruple", "large", "small", "at 1", "random", "all exponents"])
def test_logarithm(call, x):
    assert ulps(call(LOG, x), np.log(x.astype(np.longdouble))).max() <= 1.6


def test_logarithm_outside_its_range(call):
    x = np.array([0.0, -0.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 2.2e-308, 2.2250738585072014e-308, 1.7976931348623157e308])
    with np.errstate(all="ignore"):
        ref = np.log(x.astype(np.longdouble))
    got = call(LOG, x)
    ok = np.isfinite(ref)
    assert ulps(got[ok], ref[ok]).max() <= 1.6 and np.array_equal(got[~ok], ref[~ok].astype(np.float64), equal_nan=True)


@pytest.mark.parametrize("x", [
    RNG.uniform(-3.0, 3.0, 200000), RNG.uniform(-599.99, 599.99, 100000), near(np.concatenate([[600.0, -600.0], np.log(2.0) / 256 * np.arange(-301, 302, 2)])),
    spread(RNG, 50000, -60, 0) * RNG.choice([-1.0, 1.0], 50000),
], ids=["small", "range", "edges", "towards 0"])
def test_exponential(call, x):
    x = x[np.abs(x) < 600.0]
    assert ulps(call(EXP, x), np.exp(x.astype(np.longdouble))).max() <= 0.52


def test_exponential_outside_its_range(call):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 600.0, -600.0, 709.7, 710.0, -708.0, -740.0, -750.0, 1e300, -1e300])
    with np.errstate(all="ignore"):
        ref = np.exp(x)
    got = call(EXP, x)
    ok = np.isfinite(ref)
    assert np.array_equal(got[~ok], ref[~ok], equal_nan=True) and got[0] == 1.0 and got[1] == 1.0
    assert (np.abs(got[ok] - ref[ok]) <= 2.0 * np.spacing(ref[ok])).all()  # an ulp of each


def test_reciprocal(call):
    x = np.concatenate([spread(RNG, 200000, -959, 960), EDGES, 2.0 - EDGES[EDGES < 2.0], np.ldexp(EDGES, -959), np.ldexp(EDGES, 959)])
    x *= RNG.choice([-1.0, 1.0], x.size)
    assert ulps(call(RCP, x), 1.0 / x.astype(np.longdouble)).max() <= 0.52


def test_quotients(call):
    b = spread(RNG, 200000, -959, 960)
    a = b * spread(RNG, b.size, -50, 50) * RNG.choice([-1.0, 1.0], b.size)
    a, b = a[np.isfinite(a)], b[np.isfinite(a)]
    ref = a.astype(np.longdouble) / b
    assert (np.abs(call(QUOT, a, b) - ref) <= 2.1 * 2.0 ** -53 * np.abs(ref)).all()
    assert ulps(call(DIV, a, b), ref).max() <= 0.52


def test_quotients_outside_the_reciprocals_range(call):
    b = np.array([0.0, 5e-324, 1e-310, 4e-309, 1e-300, 1e300, 1.7e308, np.inf, np.nan, -0.0, -1e-310])
    for a in (0.0, 1e-320, 1e-310, 1e-290, 1.0, 1e300, np.inf, np.nan, -1e-310):
        with np.errstate(all="ignore"):
            ref = a / b
        assert np.array_equal(call(QUOT, np.full(b.shape, a), b), ref, equal_nan=True), a
        assert np.array_equal(call(DIV, np.full(b.shape, a), b), ref, equal_nan=True), a


def test_limited_slope(call):
    a = np.concatenate([spread(RNG, 100000, -540, -500), spread(RNG, 100000, -60, 2), spread(RNG, 10000, -362, -335), spread(RNG, 1000, -1070, -1000)])
    b = a * spread(RNG, a.size, -3, 3) * RNG.choice([1.0, 1.0, -1.0], a.size)
    a, b = np.concatenate([a, [1e-155, 7e-155, 2e-162, 0.0, np.nan, 1.0]]), np.concatenate([b, [1e-155, 7e-155, 3e-162, 1.0, 1.0, np.nan]])
    with np.errstate(all="ignore"):
        ref = np.where(a * b > 0, a * b * (a + b) / (a * a + b * b), 0.0)
    got = call(SLOPE, a, b)
    assert np.isfinite(got).all()
    # three roundings each way and the fused sum of squares; numerators below 2^-1022 are rounded to 2^-1074, which the quotient enlarges
    with np.errstate(all="ignore"):
        tol = 8 * 2.0 ** -53 * np.abs(ref) + np.where(a * b > 0, 4 * 2.0 ** -1074 / np.maximum(a * a + b * b, 2.0 ** -1074), 0.0)
        tol += np.where((a * b > 0) & (a * b < 2.0 ** -1022), 4 * np.abs(a + b) * 2.0 ** -1074 / np.maximum(a * a + b * b, 2.0 ** -1074), 0.0)
    assert (np.abs(got - ref) <= tol).all()


def test_sign_tests_are_comparisons(call):
    x = np.array([0.0, -0.0, 5e-324, -5e-324, 1.0, -1.0, 1.7e308, -1.7e308, np.inf, -np.inf, np.nan, np.copysign(np.nan, -1.0)])
    assert np.array_equal(call(SIGN, x), 1.0 * (x > 0) + 2.0 * (x < 0))


def test_temperature(call):
    gm1 = 1.4 - 1.0
    inv_cv = 3.0 * gm1
    rho, th = RNG.uniform(0.9, 1.1, 200000), RNG.uniform(0.15, 0.25, 200000)
    s = (np.log(th) - gm1 * np.log(rho)) / inv_cv
    ref = np.exp(np.longdouble(gm1) * np.log(rho.astype(np.longdouble)) + s.astype(np.longdouble) * inv_cv)
    assert (np.abs(call(THETA, rho, s, gm1, inv_cv) - ref) <= 4e-16 * ref).all()
