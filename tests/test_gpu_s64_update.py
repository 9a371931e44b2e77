"""The FP64-state update of the vector-record stage kernel (JZ_P32_S64) at the
sizes where its tiles, k-chunks and its widening of the increments can go
wrong, against the FP64 kernel on the same state."""
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


@pytest.mark.parametrize("shape", [(3, 3, 3), (16, 17, 18), (17, 33, 5), (34, 19, 1), (50, 16, 40)])
@pytest.mark.parametrize("kc", [None, 1, 3])
def test_update_adds_fp32_increments_to_the_fp64_state(jz, shape, kc):
    """Three steps at a fixed time step of 1e-3 on a periodic mapped box.  The
    increments of a step are a few 1e-3 of the state and carry the FP32 error
    of the fluxes, at most 1e-4 of themselves: 1e-6 of the largest value is a
    bound with room, and below what an FP32 state would leave in the
    increments.  The chunk length does not change a bit."""
    ni, nj, nk = shape
    out = {}
    for prec in (W.P64, W.P32_S64):
        grid = W.periodic_grid(ni, nj, nk, hi=(2.0, 1.5, 1.2), map_amp=0.1, map_seed=5, precision=prec)
        g = jz.Grid(grid).init(W.jet_flow(re=2e3), 0)
        g.upload(ST.random_state((nk, nj, ni), seed=11))
        if kc is not None and prec == W.P32_S64:
            jz.jz_set_tiling(g.h, kc)
        g.nsteps(3, dt=1e-3)
        out[prec] = g.download()
        g.close()
    for v in range(5):
        ref = out[W.P64][v]
        assert np.abs(out[W.P32_S64][v] - ref).max() <= 1e-6 * max(1.0, np.abs(ref).max()), v

