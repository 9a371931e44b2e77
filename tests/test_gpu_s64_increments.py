"""JZ_P32_S64: what a step adds to the FP64 state, at time steps whose
increments an FP32 state would lose."""
import numpy as np
import pytest

from paper_2003_09926_gb300 import workloads as W

import states as ST

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def jz():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_09926_gb300 import build, jz as J
    build.build()
    J.lib()
    return J


def _step(jz, shape, prec, dt, kc=None, steps=1):
    """(state before, state after) of a periodic mapped box, every node updated."""
    ni, nj, nk = shape
    grid = W.periodic_grid(ni, nj, nk, hi=(2.0, 1.5, 1.2), map_amp=0.1, map_seed=5, precision=prec)
    g = jz.Grid(grid).init(W.jet_flow(re=2e3), 0)
    g.upload(ST.random_state((nk, nj, ni), seed=11))
    if kc is not None:
        jz.jz_set_tiling(g.h, kc)
    before = g.download()
    g.nsteps(steps, dt=dt)
    after = g.download()
    g.close()
    return before, after


SHAPES = [(16, 17, 18), (17, 33, 5), (50, 16, 40)]


@pytest.mark.parametrize("shape", SHAPES)
def test_increments_below_the_fp32_spacing(jz, shape):
    """A step of 1e-9 changes the state by a few 1e-9, a hundredth of the FP32
    spacing.  The increments carry the FP32 error of the fluxes, at most 1e-4 of
    the largest increment; an FP32 state either stays or moves by a spacing."""
    a, b = _step(jz, shape, W.P64, 1e-9)
    want = b - a
    errors = {}
    for prec in (W.P32_S64, W.P32):
        a, b = _step(jz, shape, prec, 1e-9)
        errors[prec] = [np.abs((b - a)[v] - want[v]).max() / np.abs(want[v]).max() for v in range(5)]
    assert max(errors[W.P32_S64]) <= 1e-4, errors
    assert min(errors[W.P32]) >= 1e-2, errors


@pytest.mark.parametrize("shape", SHAPES + [(3, 3, 3), (34, 19, 1)])
def test_chunk_length_does_not_change_a_bit(jz, shape):
    want = _step(jz, shape, W.P32_S64, 1e-3, steps=3)[1]
    for kc in (1, 2, 3, shape[2]):
        np.testing.assert_array_equal(_step(jz, shape, W.P32_S64, 1e-3, kc, steps=3)[1], want)


def test_subnormal_increments(jz):
    """A step of 1e-38: the increments are subnormal FP32 numbers or not far above,
    which leave a state of order one as it is."""
    a, b = _step(jz, (17, 20, 9), W.P32_S64, 1e-38)
    np.testing.assert_array_equal(a, b)
