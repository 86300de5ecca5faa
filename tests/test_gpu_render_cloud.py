"""render() and gs_render_cloud: pairs that do and do not fit the first capacity, with the forward
queued before (up to 2^25 voxels) and after the count is known, against the separate calls."""
import pytest

from helpers import cloud_params, to_dev
from paper_2603_09621_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,n", [((37, 29, 21), 700), ((512, 512, 136), 300), ((16, 16, 16), 0)])
@pytest.mark.parametrize("capacity", [None, 10, 100_000])
@pytest.mark.parametrize("side", [False, True])
def test_render_equals_separate_calls(dims, n, capacity, side):
    import torch
    from paper_2603_09621_gb300 import gs
    grid, cfg = gs.Grid(*dims), gs.Config()
    d = inputs.gaussian_cloud(4, max(n, 1), dims[::-1])
    p = to_dev(cloud_params(d))[:n].contiguous()
    stream = torch.cuda.Stream() if side else None
    if side:
        stream.wait_stream(torch.cuda.current_stream())
    stats = torch.zeros(2, dtype=torch.int64, device="cuda")
    I, W, bins, ws = gs.render(p, grid, cfg, capacity, stats, stream)
    torch.cuda.synchronize()
    b2, w2 = gs.Bins(n, 100_000, grid, cfg), gs.Workspace(n, 100_000, grid, cfg)
    gs.gs_bin_bricks(p, grid, cfg, b2, w2)
    s2 = torch.zeros(2, dtype=torch.int64, device="cuda")
    I2, W2 = gs.gs_render_fwd(b2, grid, cfg, stats=s2)
    assert torch.equal(I, I2) and torch.equal(W, W2) and torch.equal(stats, s2)
    assert bins.npairs() == b2.npairs() <= bins.capacity and bins.status() == 0
    if capacity == 100_000:
        assert bins.capacity == capacity


def test_render_cloud_reports_overflow_and_bad_arguments():
    import ctypes

    import torch
    from paper_2603_09621_gb300 import gs
    grid, cfg = gs.Grid(32, 32, 32), gs.Config()
    p = to_dev(cloud_params(inputs.gaussian_cloud(4, 500, (32, 32, 32))))
    bins, ws = gs.Bins(500, 100, grid, cfg), gs.Workspace(500, 100, grid, cfg)
    I, W = torch.empty(grid.shape, device="cuda"), torch.empty(grid.shape, device="cuda")
    assert gs.gs_render_cloud(p, grid, cfg, bins, ws, I, W) == bins.npairs() > 100
    assert bins.status() == gs.GS_STATUS_CAPACITY
    g, c = grid.c(), cfg.c()
    assert gs.load().gs_render_cloud(None, ctypes.byref(g), ctypes.byref(c), ctypes.byref(bins.c), None, 0,
                                     None, None, None, None, None) == -1
    with pytest.raises(gs.GsError):
        gs.gs_render_cloud(p, gs.Grid(64, 32, 32), cfg, bins, ws, I, W)
