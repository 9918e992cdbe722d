"""The node update's own reciprocal and square roots against CUDA's correctly
rounded functions."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1701_00702_gb300 import build

pytestmark = pytest.mark.gpu
RCP, SQRT, SQRT_POS = 0, 1, 2


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    out = tmp_path_factory.mktemp("node_math") / "node_math.so"
    subprocess.run([build.nvcc(), *build.GENCODE, "-std=c++20", "-O3", "-shared", "-Xcompiler", "-fPIC", "-I",
                    str(build.CSRC), "-o", str(out), str(build.ROOT / "tests" / "node_math.cu")],
                   check=True, capture_output=True)
    L = ctypes.CDLL(str(out))

    def call(fn, a):
        a = np.ascontiguousarray(a)
        mine, cuda = np.empty_like(a), np.empty_like(a)
        f = L.node_math_f64 if a.dtype == np.float64 else L.node_math_f32
        ptr = [ctypes.c_void_p(x.ctypes.data) for x in (a, mine, cuda)]
        assert f(fn, a.size, *ptr) == 0
        return mine, cuda

    return call


def test_fp64_roots_of_special_values(evaluate):
    """NaN of either sign stays NaN (a NaN speed has to reach the run's flag),
    infinity stays infinity, zero and what lies below 2^-900 give zero."""
    nan = np.array([0x7ff8000000000000, 0xfff8000000000000, 0xfff8000000000001, 0x7fffffffffffffff], np.uint64).view(np.float64)
    for fn in (SQRT, SQRT_POS):
        assert np.isnan(evaluate(fn, nan)[0]).all()
        a = np.array([np.inf, 0.0, 5e-324, 2.0 ** -901, np.nextafter(2.0 ** -900, 0)])
        assert evaluate(fn, a)[0].tolist() == [np.inf, 0.0, 0.0, 0.0, 0.0]
        a = np.array([2.0 ** -900, 2.0 ** -898, 1.0, 4.0, 2.0 ** 1000])
        assert evaluate(fn, a)[0].tolist() == [2.0 ** -450, 2.0 ** -449, 1.0, 2.0, 2.0 ** 500]


def ulps(fn, a, r):
    """Distance of r from the exact 1/a or sqrt(a) in units of r's last place."""
    worst = 0.0
    for x, y, ulp in zip(a.tolist(), r.tolist(), np.spacing(r).tolist()):
        X, Y = Fraction(x), Fraction(y)
        err = (1 / X - Y) if fn == RCP else (X - Y * Y) / (2 * Y)
        worst = max(worst, abs(float(err / Fraction(ulp))))
    return worst


def samples(dtype, lo, hi, n=20000):
    """Random mantissas and exponents, powers of two and their neighbours, the
    update's own range about 1."""
    rng = np.random.default_rng(7)
    a = np.ldexp(rng.uniform(1, 2, n), rng.integers(lo, hi, n)).astype(dtype)
    two = np.ldexp(np.ones(9, dtype), [lo, -20, -3, -2, -1, 0, 1, 2, hi - 1])
    one = rng.uniform(0.5, 2, n).astype(dtype)
    return np.concatenate([a, two, np.nextafter(two, dtype(0)), np.nextafter(two, dtype(np.inf)), one])


@pytest.mark.parametrize("fn,lo,hi", [(RCP, -500, 500), (SQRT, -899, 1000), (SQRT_POS, -899, 1000)])
def test_fp64_within_a_64th_of_correct_rounding(evaluate, fn, lo, hi):
    """The neglected terms are below 2^-59 of the result, 2^-6 of its last place;
    so at most one last place from CUDA's correctly rounded function, rarely."""
    a = samples(np.float64, lo, hi)
    mine, cuda = evaluate(fn, a)
    assert ulps(fn, a, cuda) <= 0.5
    assert ulps(fn, a, mine) <= 0.5 + 2.0 ** -6
    off = np.abs(mine - cuda) / np.spacing(cuda)
    assert off.max() <= 1 and (off > 0).mean() <= 2.0 ** -5


@pytest.mark.parametrize("fn", [RCP, SQRT, SQRT_POS])
def test_fp32_within_the_instructions_errors(evaluate, fn):
    """rcp.approx: 1 ulp; sqrt.approx: 2^-23 of the result; rsqrt.approx, 2^-22.9,
    and the rounding of its product, 2^-24."""
    a = samples(np.float32, -100, 100)
    mine, cuda = evaluate(fn, a)
    assert (np.abs(mine - cuda) <= 2 * np.spacing(cuda)).all()
    if fn == RCP:
        assert ulps(fn, a, mine) <= 1.0
    else:
        exact = np.sqrt(a.astype(np.float64))
        assert (np.abs(mine - exact) / exact).max() <= (2.0 ** -23 if fn == SQRT else 2.0 ** -22.9 + 2.0 ** -24)
