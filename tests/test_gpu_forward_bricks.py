"""The forward render's forms (a quarter, half or whole warp per 4^3 footprint; whole warps throughout on grids of
few bricks) agree bit for bit, so no result depends on the brick shape or on the grid's extent."""
import pytest

from helpers import cloud_params, to_dev
from paper_2603_09621_gb300 import inputs

pytestmark = pytest.mark.gpu

BRICKS = [(8, 8, 8), (8, 8, 4), (4, 4, 4), (8, 4, 4), (4, 8, 4), (4, 4, 8), (4, 4, 12), (8, 4, 12), (16, 8, 4),
          (16, 4, 8), (4, 16, 4), (8, 4, 16)]


def _render(p, dims, brick):
    import torch
    from paper_2603_09621_gb300 import gs
    stats = torch.zeros(2, dtype=torch.int64, device="cuda")
    I, W, _, _ = gs.render(p, gs.Grid(*dims), gs.Config(brick=brick), stats=stats)
    return I, W, int(stats[0])


# 32^3: at most 512 footprints, whole warps throughout; 61 x 59 x 57: 3,600 and more; the others lie on
# the two sides of 2,432 footprints for 8^3 bricks (304 and 305 of them)
@pytest.mark.parametrize("dims", [(32, 32, 32), (61, 59, 57), (128, 152, 8), (8, 8, 2440)])
@pytest.mark.parametrize("brick", BRICKS[1:])
def test_brick_shapes_agree(dims, brick):
    import torch
    d = inputs.gaussian_cloud(7, min(dims[0] * dims[1] * dims[2] // 30, 8000), dims[::-1])
    p = to_dev(cloud_params(d))
    I0, W0, n0 = _render(p, dims, BRICKS[0])
    I, W, n = _render(p, dims, brick)
    assert torch.equal(I, I0) and torch.equal(W, W0) and n == n0 > 0


@pytest.mark.parametrize("brick", BRICKS)
def test_extended_grid_agrees(brick):
    """The same cloud on a grid of few bricks and on one twelve times as long, whose first slices are the same."""
    import torch
    p = to_dev(cloud_params(inputs.gaussian_cloud(9, 900, (16, 29, 30))))
    I0, W0, _ = _render(p, (30, 29, 16), brick)
    I, W, _ = _render(p, (30, 29, 16 * 40), brick)
    assert torch.equal(I[:16], I0) and torch.equal(W[:16], W0)


@pytest.mark.parametrize("brick", [(4, 4, 4), (8, 4, 4), (4, 8, 4), (4, 4, 8)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 200])
def test_small_brick_rounds(brick, n):
    """Lists of one brick about the edges of rounds of 64 records, against the same lists in 8^3 bricks."""
    import torch
    dims = (60, 64, 64)
    d = inputs.gaussian_cloud(n, n, (4, 4, 4), scale_range=(0.5, 1.5))
    p = to_dev(cloud_params(d))
    I0, W0, n0 = _render(p, dims, (8, 8, 8))
    I, W, m = _render(p, dims, brick)
    assert torch.equal(I, I0) and torch.equal(W, W0) and m == n0
