"""Slice profile and its adjoint at shapes far from a cube: few large planes, many small ones, planes that are
and are not whole 16-byte pieces. Bit for bit, and the time by volume, not by shape."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz,ny,nx,s", [(1, 1, 1, 1), (1000, 1, 1, 3), (70_001, 1, 1, 1), (70_001, 1, 2, 2),
                                        (1001, 4, 4, 4), (300, 5, 25, 7), (300, 4, 32, 5), (130, 16, 64, 3),
                                        (3, 1030, 1028, 2), (2, 2047, 2047, 1), (4, 1031, 1033, 4),
                                        (5, 33, 31, 5), (19, 33, 31, 6), (19, 12, 31, 8), (40, 33, 31, 13),
                                        (40, 32, 31, 19)])
def test_downsample_shapes(nz, ny, nx, s):
    import torch
    from paper_2603_09621_gb300 import gs
    gen = torch.Generator(device="cuda").manual_seed(nz + nx)
    hr = torch.randn((nz, ny, nx), generator=gen, device="cuda")
    nl = nz // s
    inv = torch.tensor(1.0 / s, dtype=torch.float32)
    lr = torch.full((nl, ny, nx), -7.0, device="cuda")
    if nl:
        gs.gs_downsample_fwd(hr, s, lr)
        ref = torch.zeros_like(lr)
        for j in range(s):
            ref += hr[j:nl * s:s]
        assert torch.equal(lr, ref * inv.item())
    back = gs.gs_downsample_bwd(lr, nz, s, torch.full_like(hr, -7.0))
    want = torch.zeros_like(hr)
    for j in range(s if nl else 0):
        want[j:nl * s:s] = lr * inv.item()
    assert torch.equal(back, want)


def _best_us(f):
    import torch
    best = 1e9
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


@pytest.mark.parametrize("shape,s", [((4, 2047, 2047), 4), ((4, 2047, 2047), 2), ((1_000_000, 4, 4), 1)])
def test_downsample_time_follows_the_volume(shape, s):
    """No more than three times what a volume of ordinary shape with as many voxels takes (once: 7 and 5
    times for four large planes of odd size; 4 and more for many small ones)."""
    import torch
    from paper_2603_09621_gb300 import gs
    ordinary = (64, 512, 512)

    def both(shape):
        hr = torch.zeros(shape, device="cuda")
        lr = gs.gs_downsample_fwd(hr, s)
        return _best_us(lambda: gs.gs_downsample_fwd(hr, s, lr))
    assert both(shape) < 3 * both(ordinary)
