"""Cylinders with more azimuthal points than the FP32 centreline mean holds in
registers (48 for each of its 8 warps): 384, one pair more, and two loads more."""
import numpy as np
import pytest

from paper_2003_09926_gb300 import workloads as W
from test_gpu_cyl import check_centreline_sequential

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


@pytest.mark.parametrize("prec", [W.P32, W.P32_M64])
@pytest.mark.parametrize("points", [384, 386, 390, 770])
def test_centreline_of_a_long_azimuth(jz, prec, points):
    import torch
    stream = torch.cuda.Stream()
    grid = W.cyl_grid(35, 5, points + 1, precision=prec)
    flow = W.jet_flow(re=2e4)
    alone, in_batch = (jz.Grid(grid, stream=stream).init(flow, 3) for _ in range(2))
    Q = alone.download()
    rng = np.random.default_rng(points)
    Q[1:4, :points, 1, 4] = rng.uniform(-1, 1, (3, points)) * 2.0 ** rng.integers(-30, 30, (3, points))  # not exact in integers
    Q[2, :points, 1, 5] = np.where(np.arange(points) % 2 == 0, 0.75, -0.75)
    Q[:, points] = Q[:, 0]
    alone.upload(Q)
    check_centreline_sequential(alone.download(), grid, prec)
    b = jz.Batch([in_batch], stream=stream)
    b.nsteps(2, cfl=0.5)
    alone.init(flow, 3)
    alone.nsteps(2, cfl=0.5)
    stream.synchronize()
    got = alone.download()
    check_centreline_sequential(got, grid, prec)
    np.testing.assert_array_equal(in_batch.download(), got)
    b.close()
