"""The autotuner also times what the library chooses by itself, so that its
choice is no worse than leaving a grid or a batch alone."""
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
def test_batch_choice_can_be_the_chosen_lengths(jz, monkeypatch, prec):
    import torch
    from paper_2003_09926_gb300 import autotune
    cases = [(W.jet_grid(35, 18, 16, precision=prec), W.jet_flow()),
             (W.jet_grid(67, 40, 24, precision=prec), W.jet_flow(mach=1.6))]
    ticks = iter(range(1, 1000))  # the first candidate of all is the fastest
    monkeypatch.setattr(autotune, "_time_ms", lambda *a: float(next(ticks)))
    choice = autotune.tune_batch(cases)
    assert choice["kc"] == autotune.CHOSEN
    stream = torch.cuda.Stream()
    grids = [jz.Grid(d, stream=stream).init(f, 3) for d, f in cases]
    before = [jz.jz_get_tiling(g.h) for g in grids]
    size = jz.Batch(grids, stream=stream).buf.numel()
    shape = dict(choice, shape=None)  # the lengths alone: nothing of the grids is set
    for g in grids:
        autotune.apply(g, shape)
    assert [jz.jz_get_tiling(g.h) for g in grids] == before
    assert jz.Batch(grids, stream=stream).buf.numel() == size  # the same work items


def test_grid_candidates_include_its_default(jz, monkeypatch):
    from paper_2003_09926_gb300 import autotune
    grid = W.jet_grid(69, 47, 46)
    want = jz.jz_get_tiling(jz.Grid(grid).h)[2]
    ticks = iter(range(1, 1000))
    monkeypatch.setattr(autotune, "_time_ms", lambda *a: float(next(ticks)))
    assert autotune.tune_grid(grid, W.jet_flow())["kc"] == want
    # and the real choice is of a length that runs
    monkeypatch.undo()
    autotune._cache.clear()
    assert autotune.tune_grid(W.jet_grid(40, 20, 18), W.jet_flow(), reps=1)["kc"] >= 1
