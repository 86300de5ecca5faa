"""Gradients with a truncation radius so large that it cuts nothing off: the row intervals' squared
half-widths overflow FP32 there."""
import numpy as np
import pytest

from helpers import cloud_params, to_dev
from paper_2603_09621_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("brick", [(8, 8, 8), (8, 8, 4), (4, 4, 8)])
@pytest.mark.parametrize("trunc", [1e16, 1e18, 1e19])
def test_gradient_without_truncation(trunc, brick):
    """Scales of 2-60 voxels on a 24 x 20 x 16 grid: every voxel lies within 25 sigma of every mean, so
    radii of 25, 10^16 and more include the same pairs and give the same sums."""
    import torch
    from paper_2603_09621_gb300 import gs
    grid = gs.Grid(24, 20, 16)
    d = inputs.gaussian_cloud(5, 120, grid.shape)
    d["log_s"] = np.linspace(np.log(2.0), np.log(60.0), 360).reshape(120, 3).astype(np.float32)
    p = to_dev(cloud_params(d))
    dI = torch.randn(grid.shape, generator=torch.Generator().manual_seed(1)).cuda()
    out = []
    for t in (25.0, trunc):
        cfg = gs.Config(brick=brick, trunc_sigma=t)
        I, W, bins, ws = gs.render(p, grid, cfg)
        out.append((I, W, gs.gs_render_bwd(p, bins, grid, cfg, I, W, dI, ws)))
    assert float(out[0][2].abs().max()) > 0
    for a, b in zip(*out):
        assert torch.equal(a, b)
