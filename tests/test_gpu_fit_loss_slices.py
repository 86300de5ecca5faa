"""The fitting step's loss stage at every rule of its dispatch (one kernel up to four slices per LR slice, and from
eight on for large aligned volumes; else three kernels), against the separate entry points bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,s", [((61, 45, 37), 16), ((61, 45, 37), 8), ((33, 33, 64), 5), ((16, 12, 37), 37),
                                    ((5, 3, 40), 9), ((16, 16, 33), 6), ((256, 256, 19), 9), ((256, 256, 17), 8),
                                    ((256, 256, 16), 16), ((255, 257, 17), 8), ((256, 254, 12), 5),
                                    ((258, 128, 32), 8), ((512, 256, 9), 8)])
def test_loss_stage_equals_entry_points(dims, s):
    import torch
    from paper_2603_09621_gb300 import gs
    grid, cfg = gs.Grid(*dims), gs.Config(t_act=1)
    gen = torch.Generator(device="cuda").manual_seed(s)
    n = 300
    p = torch.zeros(n, 12, device="cuda")
    p[:, :3] = torch.rand(n, 3, generator=gen, device="cuda") * torch.tensor(dims, device="cuda")
    p[:, 3:6], p[:, 6] = 1.2, 1.0
    p[:, 10] = torch.rand(n, generator=gen, device="cuda")
    target = torch.rand((dims[2] // s, dims[1], dims[0]), generator=gen, device="cuda")
    f = gs.FitState(p, target, grid, s, cfg)
    f.grad_step()
    lr = gs.gs_downsample_fwd(f.I, s)
    dpred = torch.empty_like(lr)
    loss = gs.gs_l1_loss(lr, target, f.ws, dpred=dpred)
    assert torch.equal(f.lr_pred, dpred) and torch.equal(f.d_loss, loss)
    dI = gs.gs_downsample_bwd(dpred, dims[2], s)
    grad = gs.gs_render_bwd(p, f.bins, grid, cfg, f.I, f.W, dI, f.ws)
    assert torch.equal(f.grad, grad) and grad.abs().max() > 0
    g = gs.FitState(p, target, grid, s, cfg)
    g.step()
    assert g.d_step.item() == 1 and torch.equal(g.d_loss, loss) and not torch.equal(g.params, p)
