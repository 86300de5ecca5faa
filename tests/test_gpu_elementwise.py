"""Vector and scalar forms of the volume and Adam kernels: ragged planes, trailing slices, slices
beyond the HR depth, values at 4- but not 16-byte alignment, against plain torch in 64 bits and
against each other (both forms round alike: bit for bit)."""
import pytest

pytestmark = pytest.mark.gpu


def _rand(*shape, off=0):
    """Standard normal float32 tensor whose data starts `off` floats after a 16-byte boundary."""
    import torch
    n = 1
    for s in shape:
        n *= s
    return torch.randn(n + 4, device="cuda")[off:off + n].view(shape)


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("nz,ny,nx,s", [(8, 4, 8, 4), (9, 5, 7, 2), (7, 6, 10, 3), (3, 5, 4, 5), (65, 1, 3, 1)])
def test_downsample_forms(nz, ny, nx, s, off):
    import torch
    from paper_2603_09621_gb300 import gs
    hr = _rand(nz, ny, nx, off=off)
    k = nz // s
    if k:
        lr = gs.gs_downsample_fwd(hr, s, _rand(k, ny, nx, off=off))
        ref = hr[:k * s].double().view(k, s, ny, nx).mean(1)
        assert (lr.double() - ref).abs().max() <= 2.0 ** -23 * s * hr.abs().max()  # s additions
    dlr = _rand(max(k, 1), ny, nx, off=off)
    dhr = gs.gs_downsample_bwd(dlr, nz, s, _rand(nz, ny, nx, off=off))
    want = torch.zeros_like(dhr)
    if k:
        want[:k * s] = (dlr[:k] * torch.tensor(1.0 / s, device="cuda")).repeat_interleave(s, 0)
    assert torch.equal(dhr, want)


@pytest.mark.parametrize("n", [1, 2, 85, 86, 1000])
def test_adam_forms(n):
    import torch
    from paper_2603_09621_gb300 import gs
    hp = gs.Adam()
    lr = torch.tensor([1e-3] * 3 + [5e-3] * 9, device="cuda", dtype=torch.float64)
    got = []
    for off in (0, 1):
        torch.manual_seed(n)
        p, g, m = (_rand(n, 12) for _ in range(3))
        v = _rand(n, 12) ** 2
        pp, gg, mm, vv = (_rand(n, 12, off=off).copy_(t) for t in (p, g, m, v))
        step = torch.full((), 7, dtype=torch.int32, device="cuda")
        gs.gs_adam_step(pp, gg, mm, vv, hp, step)
        assert step.item() == 8
        m64 = 0.9 * m.double() + 0.1 * g.double()
        v64 = 0.999 * v.double() + 0.001 * g.double() ** 2
        want = p.double() - lr * (m64 / (1 - 0.9 ** 8)) / ((v64 / (1 - 0.999 ** 8)).sqrt() + 1e-8)
        # p rounds once; the update (at most lr |m| / bc1 / sqrt(0.001 g^2 / bc2)) carries about ten
        # roundings of 2^-24 and a bias correction of 2^-22
        tol = 2.0 ** -24 * p.double().abs() + 2.0 ** -20 * (want - p.double()).abs() + 1e-12
        assert ((pp.double() - want).abs() <= tol).all()
        got.append((pp.clone(), mm.clone(), vv.clone()))
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("dims", [(13, 11, 10), (16, 8, 8), (5, 3, 1)])
def test_adjoint_factor_forms(dims):
    """dL/dparams with I, W, dL/dI at 16- and at 4-byte alignment, voxel counts of every remainder."""
    import torch
    from paper_2603_09621_gb300 import gs
    grid, cfg = gs.Grid(*dims), gs.Config()
    torch.manual_seed(3)
    p = torch.zeros(40, 12, device="cuda")
    p[:, :3] = torch.rand(40, 3, device="cuda") * torch.tensor(dims, device="cuda")
    p[:, 6] = 1.0
    p[:, 10:] = 0.5 + 0.2 * torch.rand(40, 2, device="cuda")
    I, W, bins, ws = gs.render(p, grid, cfg)
    dI = torch.randn_like(I)
    a = gs.gs_render_bwd(p, bins, grid, cfg, I, W, dI, ws)
    b = gs.gs_render_bwd(p, bins, grid, cfg, *(_rand(*I.shape, off=1).copy_(t) for t in (I, W, dI)), ws)
    assert torch.equal(a, b) and a.abs().max() > 0
