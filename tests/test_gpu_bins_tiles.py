"""Brick lists where the binning's tiles can go wrong, bit for bit against the oracle's
specification: Gaussian tiles of 64 and 256, rounds of 2,304 and 2,048 pairs per tile, boxes of more than 64 bricks
(counted by rows and emitted by a warp), digit widths from one narrow pass to three passes."""
import numpy as np
import pytest

from helpers import cloud_params
from paper_2603_09621_gb300 import inputs
from test_gpu_bins import _bin

pytestmark = pytest.mark.gpu

def _check(params, og, brick=(8, 8, 8)):
    import oracle
    ref = oracle.brick_lists(params, og, oracle.Config(brick=brick))
    P = ref["pair_gid"].size
    bins = _bin(params, og, brick, capacity=P + 1)
    assert bins.npairs() == P and bins.status() == 0
    for name, got in (("brick_off", bins.brick_off()), ("pair_gid", bins.pair_gid(P)), ("gm_off", bins.gm_off())):
        np.testing.assert_array_equal(got.cpu().numpy(), ref[name])
    bm_brick = np.repeat(np.arange(ref["brick_off"].size - 1), np.diff(ref["brick_off"]))
    np.testing.assert_array_equal(bins.pair_brick(P).cpu().numpy(), bm_brick)
    gmj = bins.pair_gmj(P).cpu().numpy()
    assert np.array_equal(np.sort(gmj), np.arange(P))
    np.testing.assert_array_equal(ref["gm_brick"][gmj], bm_brick)


# grid (x, y, z) and brick: 1 brick; 2 x 2 x 2; 315 (one 9-bit pass); 512 (one full pass);
# 513 x 1 x 1 (two passes, rows longer than their 32 digits); 4,096, 131,072 and 262,144 (two passes of 6, of
# 9 and 8, of 9 bits); 266,240 (three passes, of 6, 6 and 7 bits)
GRIDS = [((8, 8, 8), (8, 8, 8)), ((13, 11, 10), (8, 8, 8)), ((50, 33, 71), (8, 8, 8)),
         ((64, 64, 64), (8, 8, 8)), ((4104, 8, 8), (8, 8, 8)), ((64, 64, 64), (4, 4, 4)),
         ((512, 512, 256), (8, 8, 8)), ((512, 512, 64), (4, 4, 4)), ((520, 512, 64), (4, 4, 4))]


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1500])
@pytest.mark.parametrize("dims,brick", GRIDS)
def test_bins_tiles(dims, brick, n):
    import oracle
    og = oracle.Grid(*dims)
    d = inputs.gaussian_cloud(n + dims[0], n, dims[::-1])
    # a few wide Gaussians: boxes of tens to thousands of bricks, some clipped by the grid, next to
    # narrow ones in the same warp
    wide = np.arange(0, n, 97)
    d["log_s"][wide] += np.log(np.linspace(3.0, 12.0, wide.size))[:, None].astype(np.float32)
    _check(cloud_params(d), og, brick)


@pytest.mark.parametrize("n", [38_911, 38_912, 38_913, 39_169])
@pytest.mark.parametrize("dims,brick", [((13, 11, 10), (8, 8, 8)), ((64, 64, 64), (8, 8, 8)),
                                        ((72, 64, 64), (8, 8, 8)), ((64, 64, 60), (4, 4, 4))])
def test_bins_tile_sizes(dims, brick, n):
    """The largest cloud in tiles of 64 Gaussians and the smallest in tiles of 256, at the edges of their
    tiles, with one pass (offsets written by it) and two."""
    import oracle
    og = oracle.Grid(*dims)
    d = inputs.gaussian_cloud(n, n, dims[::-1], scale_range=(0.5, 1.2))
    d["log_s"][::4001] += 2.0
    _check(cloud_params(d), og, brick)


@pytest.mark.parametrize("n", [399_999, 400_000, 401_234])
@pytest.mark.parametrize("dims,brick", [((64, 64, 60), (4, 4, 4)), ((160, 128, 88), (8, 8, 8)),
                                        ((512, 512, 256), (8, 8, 8)), ((520, 512, 64), (4, 4, 4))])
def test_bins_count_kernel(dims, brick, n):
    """The largest cloud whose later digits are counted by the scatter before and the smallest whose
    are counted by a kernel: digits of 6 and 6, 6 and 6 of 3,520, 9 and 8, and 6, 6 and 7 bits."""
    import oracle
    og = oracle.Grid(*dims)
    d = inputs.gaussian_cloud(n, n, dims[::-1], scale_range=(0.3, 0.7))
    d["log_s"][::40_001] += 2.0
    _check(cloud_params(d), og, brick)


@pytest.mark.parametrize("h", [(1.0, 1.0, 1.0), (0.5, 2.0, 0.25), (0.9, 1.0, 1.3), (2.0 ** -8, 3.0, 4.0)])
def test_bins_voxel_sizes(h):
    """Voxel sizes that are and are not powers of two (a product and a division), offset origin."""
    import oracle
    og = oracle.Grid(53, 41, 37, h, (-3.1, 2.5, 0.7))
    d = inputs.gaussian_cloud(8, 5000, (37, 41, 53), h=h)
    d["mu"] = (d["mu"] + np.array(og.origin)).astype(np.float32)
    _check(cloud_params(d), og)


def test_bins_rounds_exact_fill():
    """Tiles of exactly 2,048 and 4,096 pairs, and one more: 256 Gaussians that all meet the same
    8 (16) bricks, plus one."""
    import oracle
    og = oracle.Grid(16, 16, 32)
    for z, n in ((8.0, 256), (8.0, 257), (16.0, 256), (16.0, 513)):
        p = np.zeros((n, 12), np.float32)
        p[:, :3] = (8.0, 8.0, z)
        p[:, 3:6] = np.log(2.0) if z == 8.0 else np.log(np.array([2.0, 2.0, 4.0]))
        p[:, 6], p[:, 10:] = 1.0, 0.5
        _check(p, og)


@pytest.mark.parametrize("nz,per", [(8, 9), (16, 18)])
@pytest.mark.parametrize("n", [38_912, 38_913, 39_167])
def test_bins_first_pass_rounds(nz, per, n):
    """First-pass tiles of 256 Gaussians (clouds of more than 38,912) and of 64 that fill rounds of 2,304
    pairs exactly, once and twice: every Gaussian meets the same 9 (18) bricks; the last tile is ragged."""
    import oracle
    p = np.zeros((n, 12), np.float32)
    p[:, :3] = (12.0, 12.0, nz / 2)
    p[:, 3:6] = np.log(np.array([2.0, 2.0, nz / 8.0]))
    p[:, 6], p[:, 10:] = 1.0, 0.5
    og = oracle.Grid(24, 24, nz)
    assert oracle.brick_lists(p, og, oracle.Config())["pair_gid"].size == per * n
    _check(p, og)


def test_bins_overflow_with_wide_gaussians():
    """Every Gaussian covers the whole grid: the count is exact, nothing is listed."""
    params = np.zeros((700, 12), np.float32)
    params[:, :3], params[:, 3:6], params[:, 6], params[:, 10:] = 100.0, 8.0, 1.0, 0.5
    import oracle
    bins = _bin(params, oracle.Grid(200, 160, 120), capacity=5000)
    assert bins.npairs() == 700 * 25 * 20 * 15 and bins.status() == 1
    assert int(bins.brick_off().abs().sum().item()) == 0
