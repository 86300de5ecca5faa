"""The fitting step's fused loss stage (slice profile, L1, adjoint factors in one kernel) against the
separate entry points, bit for bit: slice factors with and without a compiled copy, trailing
slices, odd planes (4-byte accesses), fewer LR values than one block sums, and the step counter."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(8, 8, 8), (16, 12, 23), (13, 11, 23), (5, 3, 7), (64, 48, 40)])
@pytest.mark.parametrize("s", [1, 2, 3, 4, 5, 7])
def test_fused_loss_equals_entry_points(dims, s):
    import torch
    from paper_2603_09621_gb300 import gs
    nx, ny, nz = dims
    grid, cfg = gs.Grid(*dims), gs.Config(t_act=1)
    torch.manual_seed(7 * s + nx)
    n = max(4, nx * ny * nz // 20)
    p = torch.zeros(n, 12, device="cuda")
    p[:, :3] = torch.rand(n, 3, device="cuda") * torch.tensor(dims, device="cuda")
    p[:, 3:6] = 0.3 * torch.randn(n, 3, device="cuda")
    p[:, 6] = 1.0
    p[:, 7:10] = 0.2 * torch.randn(n, 3, device="cuda")
    p[:, 10] = torch.rand(n, device="cuda")
    target = torch.rand(nz // s, ny, nx, device="cuda")
    f = gs.FitState(p, target, grid, s, cfg)
    f.grad_step()
    lr = gs.gs_downsample_fwd(f.I, s)
    dpred = torch.empty_like(lr)
    loss = gs.gs_l1_loss(lr, target, f.ws, dpred=dpred)
    assert torch.equal(f.lr_pred, dpred) and torch.equal(f.d_loss, loss)
    dI = gs.gs_downsample_bwd(dpred, nz, s)
    grad = gs.gs_render_bwd(p, f.bins, grid, cfg, f.I, f.W, dI, f.ws)
    assert torch.equal(f.grad, grad) and grad.abs().max() > 0
    assert f.d_step.item() == 0
    ref = (lr.double() - target.double()).abs().mean().item()
    assert abs(loss.item() - ref) <= 1e-6 * ref
    g = gs.FitState(p, target, grid, s, cfg)
    g.step()
    f.apply()
    assert g.d_step.item() == 1 and f.d_step.item() == 1
    for a, b in ((f.params, g.params), (f.m, g.m), (f.v, g.v)):
        assert torch.equal(a, b)
