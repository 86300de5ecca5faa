"""What render() and GaussianRender allocate, and hold between forward and backward."""
import ctypes

import pytest

from helpers import cloud_params, to_dev
from paper_2603_09621_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,n,most", [((64, 64, 32), 6000, 64 * 6000), ((32, 32, 32), 4096, 4096 * 64),
                                         ((24, 16, 8), 16_384, 16_384 * 6), ((9, 8, 8), 300, 1024),
                                         ((64, 64, 64), 40_000, 1 << 20), ((64, 64, 64), 100_000, 1_600_000)])
def test_first_capacity(dims, n, most):
    """16 pairs per Gaussian, up to 64 for small clouds, and never more than all bricks for each."""
    import torch
    from paper_2603_09621_gb300 import gs
    p = torch.zeros((n, 12), device="cuda")
    p[:, 3:6], p[:, 6] = -20.0, 1.0   # points on the volume's corner: a pair or none each
    assert gs.render(p, gs.Grid(*dims))[2].capacity == most


@pytest.mark.parametrize("dims,n", [((64, 64, 32), 6000), ((48, 48, 48), 16_384), ((16, 16, 16), 3000)])
def test_autograd_holds_no_more_than_16_pairs_per_gaussian(dims, n):
    """Between forward and backward a call holds no more than bins and scratch for 16 pairs per Gaussian, and the
    backward pass equals the separate entry points, also when it is run twice."""
    import torch
    from paper_2603_09621_gb300 import gs
    grid, cfg = gs.Grid(*dims), gs.Config()
    p = to_dev(cloud_params(inputs.gaussian_cloud(2, n, grid.shape, scale_range=(0.5, 1.5)))).requires_grad_()
    dI = torch.randn(grid.shape, generator=torch.Generator().manual_seed(1)).cuda()
    lib, g, c = gs.load(), grid.c(), cfg.c()
    most = sum(f(n, max(1024, 16 * n), ctypes.byref(g), ctypes.byref(c))
               for f in (lib.gs_bins_bytes, lib.gs_workspace_bytes)) + 2 * 4 * dI.numel() + 4 * 2**20
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    I = gs.GaussianRender.apply(p, grid, cfg)
    assert torch.cuda.memory_allocated() - before <= most
    g1, = torch.autograd.grad(I, p, dI, retain_graph=True)
    g2, = torch.autograd.grad(I, p, dI)
    I3, W3, bins, ws = gs.render(p.detach(), grid, cfg)
    g3 = gs.gs_render_bwd(p.detach(), bins, grid, cfg, I3, W3, dI, ws)
    assert torch.equal(I.detach(), I3) and torch.equal(g1, g3) and torch.equal(g2, g3)
