"""The FP64 elementary functions that the FP64 kernels evaluate from the
hardware's approximations, against extended precision over mantissas and
exponents."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RCP, SQRT, JM23, JM23_LIBRARY = range(4)


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_09926_gb300 import build
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "probes", "fastmath_probe.cu")
    lib = str(tmp_path_factory.mktemp("probe") / "fastmath_probe.so")
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-o", lib, src],
                   check=True)
    fn = C.CDLL(lib).fastmath_eval
    P = C.POINTER(C.c_double)
    fn.argtypes = [C.c_int, C.c_int, P, P]

    def run(which, x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.empty_like(x)
        assert fn(which, x.size, x.ctypes.data_as(P), y.ctypes.data_as(P)) == 0
        return y

    return run


def _numbers(lo, hi, n=300_000):
    """Random mantissas, and those nearest to powers of two, at exponents lo .. hi."""
    rng = np.random.default_rng(17)
    m = 1.0 + rng.random(n)
    edge = [1.0, 1.0 + 2.0 ** -52, 1.0 + 2.0 ** -51, 2.0 - 2.0 ** -52, 2.0 - 2.0 ** -51, 1.5]
    ex = rng.integers(lo, hi + 1, n)
    every = np.arange(lo, hi + 1)
    return np.concatenate([np.ldexp(m, ex)] + [np.ldexp(v, every) for v in edge])


def _ulps(got, exact):
    """Error of got in units in the last place of the exact value."""
    unit = np.spacing(np.abs(exact.astype(np.float64))).astype(np.longdouble)
    return np.abs(got.astype(np.longdouble) - exact) / unit


# The approximations are within 2^-19 relatively, so the terms left out of
# the series are below 2^-75 and the roundings of the correction, itself
# below 2^-18 of the result, below 2^-69: 2^-16 units in the last place beside
# the last rounding's half.  J^(-2/3) also carries 2/3 of the rounding of y^3,
# at most 2/3 of a unit.


def test_reciprocal(evaluate):
    x = _numbers(-1000, 1000)
    x[::2] *= -1.0
    assert _ulps(evaluate(RCP, x), np.longdouble(1.0) / x.astype(np.longdouble)).max() <= 0.5 + 2.0 ** -10


def test_square_root(evaluate):
    x = _numbers(-1000, 1000)
    assert _ulps(evaluate(SQRT, x), np.sqrt(x.astype(np.longdouble))).max() <= 0.5 + 2.0 ** -10


def test_power_minus_two_thirds(evaluate):
    x = _numbers(-900, 900)
    c = np.cbrt(x.astype(np.longdouble))
    exact = 1.0 / (c * c)
    err, library = _ulps(evaluate(JM23, x), exact), _ulps(evaluate(JM23_LIBRARY, x), exact)
    assert err.max() <= 0.5 + 2.0 / 3.0 + 2.0 ** -10
    assert np.sqrt((err ** 2).mean()) <= np.sqrt((library ** 2).mean())
