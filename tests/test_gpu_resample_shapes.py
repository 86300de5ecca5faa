"""Trilinear resize and its adjoint at shapes far from a cube: one to a few dozen columns, more columns than 48 KB
of shared memory take, planes that no sample reads; against 64-bit sums with the FP32 positions of the definition."""
import pytest

from test_gpu_volume_shapes import _best_us

pytestmark = pytest.mark.gpu


def _axis(a, src, dst):
    import torch
    j = torch.arange(dst[a], device="cuda", dtype=torch.float32) + 0.5
    scale = torch.tensor(float(src[a]), device="cuda") / torch.tensor(float(dst[a]), device="cuda")
    c = (j * scale - 0.5).clamp_min(0.0)
    i0 = c.floor().long()
    w = (c - c.floor()).double().view([-1 if k == a else 1 for k in range(3)])
    return i0, (i0 + 1).clamp_max(src[a] - 1), w


def _fwd64(x, src, dst):
    v = x.double()
    for a in range(3):
        i0, i1, w = _axis(a, src, dst)
        v = v.index_select(a, i0) * (1 - w) + v.index_select(a, i1) * w
    return v


def _bwd64(d, src, dst):
    import torch
    v = d.double()
    for a in range(3):
        i0, i1, w = _axis(a, src, dst)
        shape = list(v.shape)
        shape[a] = src[a]
        z = torch.zeros(shape, dtype=torch.float64, device="cuda")
        v = z.index_add_(a, i0, v * (1 - w)).index_add_(a, i1, v * w)
    return v


SHAPES = ([((70, 65, n), (70, 65, n)) for n in (1, 2, 3, 4, 17, 55, 56, 57, 60)] +        # an exact copy
          [((30, 33, n), (10, 33, n)) for n in (1, 5, 20, 56, 57, 64)] +                  # planes that nothing reads
          [((31, 40, n), (13, 17, max(1, n // 3))) for n in (1, 4, 20, 56, 57, 129)] +
          [((31, 40, n), (29, 38, (n * 4 + 2) // 3)) for n in (3, 20, 56, 57)] +          # four taps
          [((90, 6, 6), (30, 2, 2)), ((27, 9, 57), (9, 3, 19)), ((200, 1, 1), (67, 1, 1)), ((1, 1, 9), (1, 1, 3)),
           ((65, 300, 1), (64, 299, 1)), ((4, 9, 512), (1, 9, 512)), ((5, 9, 700), (2, 9, 699)),
           ((3, 17, 1000), (1, 17, 1000)), ((3, 17, 1030), (1, 16, 1030)), ((3, 9, 900), (3, 9, 1300))])


@pytest.mark.parametrize("src,dst", SHAPES)
def test_resize_shapes_64bit(src, dst):
    import torch
    from paper_2603_09621_gb300 import gs
    gen = torch.Generator(device="cuda").manual_seed(sum(src))
    x, d = torch.randn(src, generator=gen, device="cuda"), torch.randn(dst, generator=gen, device="cuda")
    terms, u = 1.0, 2.0 ** -24
    for s, t in zip(src, dst):
        terms *= t / s + 3
    # forward: about ten roundings of weights and products of values up to max |x|; adjoint: the same per term
    fwd = torch.full(dst, -7.0, device="cuda")
    gs.gs_resample_fwd(x, dst, fwd)
    assert (fwd.double() - _fwd64(x, src, dst)).abs().max() <= 12 * u * x.abs().max()
    out = torch.full((x.numel() + 1,), -7.0, device="cuda")
    gs.gs_resample_bwd(d, src, out[:x.numel()])
    got = out[:x.numel()].view(src)
    assert (got.double() - _bwd64(d, src, dst)).abs().max() <= (12 + terms) * terms * u * d.abs().max()
    assert out[-1] == -7.0
    # the copy for unaligned volumes gives the same bits
    off = torch.full((x.numel() + 1,), -7.0, device="cuda")
    gs.gs_resample_bwd(d, src, off[1:])
    assert torch.equal(off[1:].view(src), got) and off[0] == -7.0


@pytest.mark.parametrize("dims,lr_shape", [((20, 24, 30), (10, 24, 20)), ((5, 33, 31), (5, 33, 31)),
                                           ((56, 34, 9), (56, 17, 3)), ((57, 34, 9), (57, 17, 3)),
                                           ((512, 8, 12), (512, 8, 4))])
def test_fused_adjoint_equals_entry_points(dims, lr_shape):
    """The fitting step's fused adjoint at these shapes, against the separate calls bit for bit."""
    from test_gpu_fit_loss import test_trilinear_step_equals_entry_points as check
    check(dims, lr_shape[::-1])


def test_resize_time_follows_the_volume():
    """2,048 x 2,048 samples of one column take no more than four times one plane of as many (once 13 times, and 8
    times for the adjoint)."""
    import torch
    from paper_2603_09621_gb300 import gs

    def both(src, dst):
        x, d = torch.zeros(src, device="cuda"), torch.zeros(dst, device="cuda")
        return (_best_us(lambda: gs.gs_resample_fwd(x, dst, d)), _best_us(lambda: gs.gs_resample_bwd(d, src, x)))
    thin, plane = both((2048, 2048, 1), (1024, 1024, 1)), both((1, 2048, 2048), (1, 1024, 1024))
    assert thin[0] < 4 * plane[0] and thin[1] < 4 * plane[1], (thin, plane)
