"""The node update's own reciprocal and square roots against CUDA's correctly
rounded functions."""
import ctypes
import subprocess

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
