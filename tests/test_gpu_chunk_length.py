"""k-chunk lengths set with jz_set_tiling beyond the grid's planes, up to the
largest integer: the whole column, alone and in a batch."""
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


@pytest.mark.parametrize("prec", [W.P64, W.P32_M64, W.P32, W.P32_S64])
@pytest.mark.parametrize("kc", [17, 2 ** 31 - 18, 2 ** 31 - 1])
def test_chunk_longer_than_the_grid(jz, prec, kc):
    import torch
    stream = torch.cuda.Stream()
    descs = [W.jet_grid(33, 20, 18, precision=prec), W.jet_grid(50, 17, 4, precision=prec)]
    flow = W.jet_flow()

    def grids():
        return [jz.Grid(d, stream=stream).init(flow, 3) for d in descs]

    want = []
    for g in grids():
        g.nsteps(2, cfl=0.5)
        want.append(g.download())
    alone, batched = grids(), grids()
    for g in alone + batched:
        jz.jz_set_tiling(g.h, kc)
        assert jz.jz_get_tiling(g.h)[2] == kc
    for g, ref in zip(alone, want):
        g.nsteps(2, cfl=0.5)
        np.testing.assert_array_equal(g.download(), ref)
    b = jz.Batch(batched, stream=stream)
    b.nsteps(2, cfl=0.5)
    stream.synchronize()
    for g, ref in zip(batched, want):
        np.testing.assert_array_equal(g.download(), ref)
    b.close()
