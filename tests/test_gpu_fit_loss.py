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


@pytest.mark.parametrize("dims,lr_shape", [((16, 12, 23), (9, 5, 7)), ((13, 11, 23), (23, 11, 13)),
                                           ((64, 70, 90), (41, 33, 64)), ((30, 34, 20), (13, 40, 32)),
                                           ((21, 19, 17), (6, 8, 10)), ((20, 16, 12), (40, 33, 7))])
def test_trilinear_step_equals_entry_points(dims, lr_shape):
    """Resize adjoint fused with the factors (aligned quads and single voxels; two-tap, four-tap and
    general runs; one and two planes per block) against gs_resample_bwd and gs_render_bwd."""
    import torch
    from paper_2603_09621_gb300 import gs
    grid, cfg = gs.Grid(*dims), gs.Config(t_act=1)
    torch.manual_seed(dims[0])
    n = 400
    p = torch.zeros(n, 12, device="cuda")
    p[:, :3] = torch.rand(n, 3, device="cuda") * torch.tensor(dims, device="cuda")
    p[:, 3:6] = 0.8
    p[:, 6] = 1.0
    p[:, 10] = torch.rand(n, device="cuda")
    target = torch.rand(lr_shape, device="cuda")
    f = gs.FitState(p, target, grid, 0, cfg, lr_model=gs.GS_LR_TRILINEAR)
    f.grad_step()
    lr = gs.gs_resample_fwd(f.I, lr_shape)
    dpred = torch.empty_like(lr)
    loss = gs.gs_l1_loss(lr, target, f.ws, dpred=dpred)
    assert torch.equal(f.lr_pred, dpred) and torch.equal(f.d_loss, loss)
    dI = gs.gs_resample_bwd(dpred, f.I.shape)
    grad = gs.gs_render_bwd(p, f.bins, grid, cfg, f.I, f.W, dI, f.ws)
    assert torch.equal(f.grad, grad) and grad.abs().max() > 0


@pytest.mark.parametrize("src,dst", [((20, 33, 41), (131, 150, 301)), ((40, 50, 64), (12, 20, 257)),
                                     ((155, 61, 43), (70, 31, 20))])
def test_resize_forms_64bit(src, dst):
    """One row and four rows per thread (from 5M destination voxels), more columns than a block has,
    forward and adjoint against 64-bit sums with the FP32 positions of the definition."""
    import torch
    from paper_2603_09621_gb300 import gs
    torch.manual_seed(1)
    x, d = torch.randn(src, device="cuda"), torch.randn(dst, device="cuda")
    fwd, bwd = x.double(), d.double()
    for a in range(3):
        j = torch.arange(dst[a], device="cuda", dtype=torch.float32) + 0.5
        scale = torch.tensor(float(src[a]), device="cuda") / torch.tensor(float(dst[a]), device="cuda")
        c = (j * scale - 0.5).clamp_min(0.0)
        i0 = c.floor().long()
        i1 = (i0 + 1).clamp_max(src[a] - 1)
        w = (c - c.floor()).double().view([-1 if k == a else 1 for k in range(3)])
        fwd = fwd.index_select(a, i0) * (1 - w) + fwd.index_select(a, i1) * w
        shape = list(bwd.shape)
        shape[a] = src[a]
        z = torch.zeros(shape, dtype=torch.float64, device="cuda")
        bwd = z.index_add_(a, i0, bwd * (1 - w)).index_add_(a, i1, bwd * w)
    # forward: about ten roundings of weights and products of values up to max |x|; adjoint: the same per
    # term, with up to (dst / src + 3)^3 terms
    terms = 1.0
    for s, t in zip(src, dst):
        terms *= t / s + 3
    u = 2.0 ** -24
    assert (gs.gs_resample_fwd(x, dst).double() - fwd).abs().max() <= 12 * u * x.abs().max()
    assert (gs.gs_resample_bwd(d, src).double() - bwd).abs().max() <= (12 + terms) * terms * u * d.abs().max()


def test_refused_step_is_not_counted():
    """Adam parameters out of range: the step is refused before anything is launched."""
    import torch
    from paper_2603_09621_gb300 import gs
    grid = gs.Grid(16, 12, 8)
    p = torch.zeros(50, 12, device="cuda")
    p[:, :3], p[:, 6] = 5.0, 1.0
    f = gs.FitState(p.clone(), torch.rand(4, 12, 16, device="cuda"), grid, 2, gs.Config(),
                    adam=gs.Adam(beta1=1.0))
    for step in (f.step, lambda: f.step_host(torch.ones(50, 12))):
        with pytest.raises(Exception, match="INVALID_ARG"):
            step()
        torch.cuda.synchronize()
        assert int(f.d_step) == 0 and torch.equal(f.params, p)
