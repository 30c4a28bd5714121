"""The float64 path's own elementary functions against long double.

Each function is evaluated on the device over its branches, with the points
around every branch's edge, and compared with numpy's long double (64 bits of
mantissa or more).  Bounds, in units in the last place of the result unless
said otherwise:

* rcp 0.52 (one third-order step: the seed's error cubed is below 2^-60),
  sqrt_ and rsqrt_ 1.0 (a rounding of x y half stays in),
* expm1 and log1p 0.75 below 1/4 and 1/8 (above, CUDA's functions bit for bit),
* unit_log 1.0; the uniforms' cosine and sine 1.4e-16 absolute (half a last
  place each for the table value and the sum, the rest below 0.3e-16),
* pair_r64 2.8e-14 relative: with d the error of H (the roundings of y, 9e-8,
  and of r^2 and the product, 6e-8 each) and g that of 1/H (2.4e-7, of the same
  sign) it is d (g - d / 2); with a second step half an ulp for r and 3e-16
  relative for 1/r.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1707_04232_gb300 import build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

FN = {k: i for i, k in enumerate(["rcp", "sqrt", "rsqrt", "expm1", "log1p", "pair_r", "pair_r2", "pair_rinv",
                                  "unit_log", "unit_cos", "unit_sin", "unit_value", "cuda_expm1", "cuda_log1p"])}
LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    here = os.path.dirname(os.path.abspath(__file__))
    so = str(tmp_path_factory.mktemp("f64") / "float64_functions.so")
    subprocess.run([build.nvcc(), build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-cudart", "shared", "-I", build.CSRC, "-I", build.INCLUDE, "-o", so,
                    os.path.join(here, "float64_functions.cu")], check=True, capture_output=True)
    out = C.CDLL(so)
    out.eval.argtypes = [C.c_int, C.c_int64, C.c_void_p, C.c_void_p]
    return out


def evaluate(lib, name, x):
    """x: float64, or uint64 (the unit functions)."""
    d = torch.from_numpy(np.ascontiguousarray(x).view(np.float64)).cuda()
    y = torch.empty_like(d)
    torch.cuda.synchronize()
    assert lib.eval(FN[name], d.numel(), d.data_ptr(), y.data_ptr()) == 0
    return y.cpu().numpy()


def ulps(got, exact):
    return np.abs((got.astype(LD) - exact) / np.spacing(np.abs(exact.astype(np.float64))).astype(LD)).max()


def spread(lo, hi, n=100_000, seed=0):
    """Logarithmically spread numbers of [lo, hi] with both ends and their neighbours."""
    x = np.exp(np.random.default_rng(seed).uniform(np.log(lo), np.log(hi), n))
    ends = [np.nextafter(e, d) for e in (lo, hi) for d in (0.0, e, np.inf)]
    return np.concatenate([np.clip(x, lo, hi), ends])


def both_signs(x):
    return np.concatenate([x, -x])


@pytest.mark.parametrize("name,ranges,bound", [
    ("expm1", [(1e-300, 1e-40), (1e-40, 2.0 ** -10), (2.0 ** -10, 2.0 ** -6), (2.0 ** -6, 0.125), (0.125, 0.25)], 0.75),
    ("log1p", [(1e-300, 1e-40), (1e-40, 2.0 ** -10), (2.0 ** -10, 2.0 ** -6), (2.0 ** -6, 0.0625), (0.0625, 0.125)], 0.75),
])
def test_expm1_and_log1p(lib, name, ranges, bound):
    for lo, hi in ranges:
        x = both_signs(spread(lo, hi))
        if (name, hi) in (("expm1", 0.25), ("log1p", 0.125)):
            x = x[np.abs(x) < hi]
        assert ulps(evaluate(lib, name, x), getattr(np, name)(x.astype(LD))) <= bound


def test_expm1_and_log1p_beyond_their_series(lib):
    for name, x in (("expm1", both_signs(spread(0.25, 30.0))), ("log1p", both_signs(spread(0.125, 0.99)))):
        x = x[np.abs(x) >= {"expm1": 0.25, "log1p": 0.125}[name]]
        assert np.array_equal(evaluate(lib, name, x), evaluate(lib, "cuda_" + name, x))


def test_reciprocal_and_roots(lib):
    x = np.concatenate([spread(1e-280, 1e280), spread(0.5, 4.0)])
    assert ulps(evaluate(lib, "rcp", both_signs(x)), 1 / both_signs(x).astype(LD)) <= 0.52
    x = np.concatenate([x, spread(2.0 ** -970, 2.0 ** -950)])  # the seed's flush range
    assert ulps(evaluate(lib, "sqrt", x), np.sqrt(x.astype(LD))) <= 1.0
    assert ulps(evaluate(lib, "rsqrt", x), 1 / np.sqrt(x.astype(LD))) <= 1.0


def test_pair_distances(lib):
    x = np.concatenate([spread(1e-12, 10.0), spread(1.0, 4.0, seed=1), spread(1e-36, 1e37),
                        spread(1e-30, 1.1e-30, n=1000)])
    r = np.sqrt(x.astype(LD))
    assert np.abs(evaluate(lib, "pair_r", x) / r - 1).max() <= 2.8e-14
    assert np.abs(evaluate(lib, "pair_r2", x) / r - 1).max() <= 2.3e-16
    assert np.abs(evaluate(lib, "pair_rinv", x) * r - 1).max() <= 3e-16


def uniforms():
    """Units of 2^-54: random words of every size, the two ends, and the
    logarithm table's interval edges (1 + j/128, j = 52, 53 and 54 among them)."""
    rng = np.random.default_rng(3)
    x = rng.integers(0, 2 ** 53, 200_000, dtype=np.uint64) >> rng.integers(0, 53, 200_000).astype(np.uint64)
    v = 2 * x + 1
    v = np.where(x >> np.uint64(52), v - 1 + (v & 2), v)
    edges = np.array([(128 + j) << 46 for j in range(129)], dtype=np.uint64)  # 2^53 (1 + j / 128)
    ends = np.array([1, 2, 3, 2 ** 54, 2 ** 54 - 2, 2 ** 53, 2 ** 53 - 1], dtype=np.uint64)
    return np.concatenate([v, edges, edges - 2, edges[:-1] + 2, ends]).astype(np.uint64)


def test_random_number_functions(lib):
    v = uniforms()
    u = v.astype(LD) * LD(2) ** -54
    assert np.array_equal(evaluate(lib, "unit_value", v), u.astype(np.float64))
    assert ulps(evaluate(lib, "unit_log", v)[v < 2 ** 54], np.log(u[v < 2 ** 54])) <= 1.0
    assert (evaluate(lib, "unit_log", v)[v == 2 ** 54] == 0.0).all()
    v = np.concatenate([v, np.arange(0, 2 ** 54 + 1, 2 ** 47, dtype=np.uint64)])  # the angles' table edges
    a = 2 * PI * (v.astype(LD) * LD(2) ** -54)
    assert np.abs(evaluate(lib, "unit_cos", v) - np.cos(a)).max() <= 1.4e-16
    assert np.abs(evaluate(lib, "unit_sin", v) - np.sin(a)).max() <= 1.4e-16
