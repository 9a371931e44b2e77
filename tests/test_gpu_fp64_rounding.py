"""Rounding errors of the FP64 kernels' building blocks, against extended
precision: the elementary functions that they evaluate from the hardware's
approximations, over mantissas and exponents, the face flux, and the widening of
the FP64-state update."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RCP, SQRT, JM23, JM23_LIBRARY, WIDEN = range(5)


P = C.POINTER(C.c_double)


def _dp(a):
    return a.ctypes.data_as(P)


def _probe(tmp_path_factory, name):
    """tests/probes/<name>.cu, which includes the kernels' source, as a library."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_09926_gb300 import build
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "probes", name + ".cu")
    lib = str(tmp_path_factory.mktemp("probe") / (name + ".so"))
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-o", lib, src],
                   check=True)
    return C.CDLL(lib)


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    fn = _probe(tmp_path_factory, "fastmath_probe").fastmath_eval
    fn.argtypes = [C.c_int, C.c_int, P, P]

    def run(which, x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.empty_like(x)
        assert fn(which, x.size, _dp(x), _dp(y)) == 0
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


@pytest.fixture(scope="module")
def face(tmp_path_factory):
    fn = _probe(tmp_path_factory, "face_probe").face_eval
    fn.argtypes = [C.c_int, C.c_double, C.c_double, P, P]
    return fn


def test_face_flux_rounds_once_at_the_size_of_the_sum(face):
    """2h = Ga + Gb - l2 d1 + l4 d3 with Ga, Gb in [1, 1.9] and a dissipation
    below 2^-10 of them.  Of the three roundings one is of the sum (in [2, 4):
    2^-52 at most) and two of Ga and Gb with their share of the dissipation
    (in [1, 2): 2^-53 each): 2^-51, and below 2^-60 from the dissipation's own
    roundings.  Adding the dissipation to the sum would round three times at
    its size, up to 1.5 2^-51."""
    n, k2, k4 = 200_000, 0.25, 2.0 ** -8
    rng = np.random.default_rng(3)
    x = np.empty((n, 34))
    x[:, :14] = 1.0 + 0.9 * rng.random((n, 14))
    x[:, [5, 12]] = 0.5 * rng.random((n, 2))  # radii
    x[:, [6, 13]] = 0.01 * rng.random((n, 2))  # sensors
    x[:, 14:] = 1.0 + 2.0 ** -6 * rng.random((n, 20))
    y = np.empty((n, 5))
    assert face(n, k2, k4, _dp(x), _dp(y)) == 0
    L = x.astype(np.longdouble)
    Ga, Gb = L[:, 0:5], L[:, 7:12]
    qm, qa, qb, qp = (L[:, 14 + 5 * m:19 + 5 * m] for m in range(4))
    lam = (L[:, 5] + L[:, 12])[:, None]
    e2 = k2 * np.maximum(L[:, 6], L[:, 13])[:, None]
    e4 = np.maximum(0.0, k4 - e2)
    exact = Ga + Gb - lam * (e2 * (qb - qa) - e4 * (qp - 3 * qb + 3 * qa - qm))
    assert np.abs(y - exact).max() <= 2.0 ** -51 * (1.0 + 2.0 ** -8)


def test_zero_infinity_and_nan(evaluate):
    """As in IEEE arithmetic, with subnormal numbers taken as zero."""
    inf, nan, tiny, big = np.inf, np.nan, 2.0 ** -1030, np.finfo(np.float64).max
    x = np.array([0.0, -0.0, inf, -inf, nan, -nan, tiny, -tiny])
    np.testing.assert_array_equal(evaluate(RCP, x), [inf, -inf, 0.0, -0.0, nan, nan, inf, -inf])
    np.testing.assert_array_equal(np.signbit(evaluate(RCP, x[2:4])), [False, True])
    x = np.array([0.0, -0.0, inf, -inf, nan, -nan, tiny, -1.0, -big])
    np.testing.assert_array_equal(evaluate(SQRT, x), [0.0, 0.0, inf, nan, nan, nan, 0.0, nan, nan])
    x = np.array([0.0, inf, nan, -nan, tiny])
    np.testing.assert_array_equal(evaluate(JM23, x), [inf, 0.0, nan, nan, inf])
    # the ends of the normal numbers
    x = np.array([2.0 ** -1022, 2.0 ** 1021, big, 2.0 ** 1023])
    np.testing.assert_allclose(evaluate(RCP, x), 1.0 / x, rtol=2.0 ** -52, atol=2.0 ** -1022)
    np.testing.assert_array_equal(evaluate(SQRT, x), np.sqrt(x))


def test_a_nan_sensor_reaches_the_face_flux(face):
    """Whichever side of a face has it, and whatever its sign: the state then
    shows it instead of going on with the other side's dissipation."""
    n = 4
    x = np.ones((n, 34))
    x[:, [6, 13]] = 0.01
    x[0, 6], x[1, 6] = np.nan, -np.nan
    x[2, 13], x[3, 13] = np.nan, -np.nan
    y = np.zeros((n, 5))
    assert face(n, 0.25, 2.0 ** -8, _dp(x), _dp(y)) == 0
    assert np.isnan(y).all()
    x[:, [6, 13]] = [[0.01, np.inf], [np.inf, 0.01], [-0.5, 0.01], [0.01, -0.5]]
    x[:, 24] = 1.5  # a density jump at the face
    assert face(n, 0.25, 2.0 ** -8, _dp(x), _dp(y)) == 0
    assert not np.isfinite(y[:2, 0]).any() and np.isfinite(y[2:]).all()


def test_increments_are_widened_exactly(evaluate):
    """Groups of five FP32 numbers of every exponent, zeros, subnormal numbers,
    infinities and NaN among them: alone in a group, and in groups of their own."""
    rng = np.random.default_rng(9)
    x = rng.integers(0, 2 ** 32, 5 * 100_000, dtype=np.uint64).astype(np.uint32).view(np.float32)
    special = np.array([0x0, 0x80000000, 0x1, 0x80000001, 0x7fffff, 0x807fffff, 0x800000, 0x80800000, 0x7f7fffff,
                        0xff7fffff, 0x7f800000, 0xff800000, 0x7fc00000, 0xffc00000, 0x3f800000], np.uint32)
    g = np.full((15, 5, 5), 1.25, np.float32)
    for k in range(5):
        g[:, k, k] = special.view(np.float32)
    x = np.concatenate([x, special.view(np.float32), g.ravel()])
    with np.errstate(invalid="ignore"):
        want = x.astype(np.float64)
    got = evaluate(WIDEN, want)
    number = ~np.isnan(want)
    np.testing.assert_array_equal(got[number].view(np.int64), want[number].view(np.int64))
    assert np.isnan(got[~number]).all()
