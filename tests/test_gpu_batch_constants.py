"""Batches whose grids share a flow model but not its constants: the stage
kernel then takes the constants of every grid from its own table entry."""
import numpy as np
import pytest

from paper_2003_09926_gb300 import workloads as W

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


@pytest.mark.parametrize("prec", [W.P32, W.P32_S64, W.P64])
@pytest.mark.parametrize("base", [dict(), dict(re=5e3, sgs=W.SGS_VREMAN), dict(re=0.0, cs=0.0)])
def test_grids_of_one_model_with_their_own_constants(jz, prec, base):
    import torch
    stream = torch.cuda.Stream()
    own = [dict(), dict(gamma=1.3), dict(cs=0.15) if base.get("cs") != 0.0 else dict(k4=0.005), dict(k2=0.3, pr=0.8)]
    shapes = [(36, 22, 18), (33, 17, 19), (20, 18, 12), (24, 20, 14)]
    cases = [(W.jet_grid(*sh, map_amp=0.03, map_seed=k, precision=prec), W.jet_flow(**{**base, **o}), 40 + k)
             for k, (sh, o) in enumerate(zip(shapes, own))]
    grids = [jz.Grid(g, stream=stream).init(f, s) for g, f, s in cases]
    b = jz.Batch(grids, stream=stream)
    b.nsteps(3, cfl=0.5)
    stream.synchronize()
    for (g, f, s), bg in zip(cases, grids):
        alone = jz.Grid(g).init(f, s)
        alone.nsteps(3, cfl=0.5)
        np.testing.assert_array_equal(bg.download(), alone.download())
        alone.close()
    b.close()
