"""A launch that CUDA refuses is reported by the call that made it, and by no
later one of this library or of another in the process."""
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


@pytest.mark.parametrize("prec", [W.P32, W.P32_M64, W.P64])
def test_a_refused_launch_leaves_no_error_behind(jz, prec):
    import torch
    # 65,998 chunks of one plane: more blocks in z than a launch may have
    g = jz.Grid(W.jet_grid(3, 3, 66000, precision=prec)).init(W.jet_flow(), 0)
    kc = jz.jz_get_tiling(g.h)[2]
    jz.jz_set_tiling(g.h, 1)
    with pytest.raises(jz.JzError) as ei:
        g.step(cfl=0.5)
    assert ei.value.code == jz.JZ_ECUDA
    torch.ones(4, device="cuda").add_(1)  # checks the last error after its launch
    jz.jz_set_tiling(g.h, max(kc, 8))
    g.init(W.jet_flow(), 0)
    g.step(dt=1e-8)
    assert g.diagnostics()["step"] == 1
    g.close()
