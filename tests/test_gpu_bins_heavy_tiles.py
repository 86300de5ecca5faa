"""Brick lists of clouds whose pairs sit in few Gaussians: a first-pass tile of more than 9,216 pairs is shared
out in parts among several blocks. Bit for bit against the oracle's specification."""
import numpy as np
import pytest

from helpers import cloud_params, to_dev
from paper_2603_09621_gb300 import inputs
from test_gpu_bins_tiles import _check

pytestmark = pytest.mark.gpu


def _cover(n, dims, sigma=2000.0):
    """n Gaussians that meet every brick of the grid."""
    p = np.zeros((n, 12), np.float32)
    p[:, :3] = np.array(dims, np.float32) / 2
    p[:, 3:6] = np.log(sigma)
    p[:, 6], p[:, 10:] = 1.0, 0.5
    return p


# bricks (digits): 512 (one pass), 4,096 (6 and 6 bits), 131,072 (9 and 8), 266,240 (6, 6 and 7)
@pytest.mark.parametrize("dims,brick,n", [((64, 64, 64), (8, 8, 8), 1), ((64, 64, 64), (8, 8, 8), 64),
                                          ((64, 64, 64), (8, 8, 8), 150), ((61, 59, 57), (4, 4, 4), 65),
                                          ((512, 512, 256), (8, 8, 8), 1), ((512, 512, 256), (8, 8, 8), 180),
                                          ((520, 512, 64), (4, 4, 4), 5)])
def test_bins_all_wide(dims, brick, n):
    """Every tile is heavy; 180 Gaussians on 131,072 bricks are 23.6M pairs, whose parts are longer than 9,216."""
    import oracle
    _check(_cover(n, dims), oracle.Grid(*dims), brick)


@pytest.mark.parametrize("dims,brick", [((64, 64, 64), (8, 8, 8)), ((64, 64, 60), (4, 4, 4)),
                                        ((520, 16, 4104), (8, 8, 8))])
@pytest.mark.parametrize("n", [300, 38_912, 38_913])
def test_bins_wide_among_narrow(dims, brick, n):
    """Wide Gaussians of many sizes, clipped by the grid, alone and in a row, in tiles of 64 and of 256."""
    import oracle
    d = inputs.gaussian_cloud(n, n, dims[::-1], scale_range=(0.5, 1.2))
    wide = np.unique(np.concatenate([np.arange(5, n, max(n // 9, 40)), np.arange(64, 96), [n - 1]]))
    d["log_s"][wide] = np.log(np.geomspace(4.0, 400.0, wide.size))[:, None].astype(np.float32)
    _check(cloud_params(d), oracle.Grid(*dims), brick)


@pytest.mark.parametrize("bricks,more", [(144, 0), (144, 1), (144, 63), (288, 0), (288, 1), (36, 0), (37, 0)])
@pytest.mark.parametrize("n", [64, 100])
def test_bins_part_edges(bricks, more, n):
    """Tiles of exactly one and two parts (64 x 144 and 64 x 288 pairs), and of one pair or a few more: on a
    row of bricks + 1 bricks, `more` of the first 64 Gaussians meet one brick more than the others."""
    import oracle
    nx = 8 * (bricks + 1)
    p = _cover(n, (nx, 8, 8))
    p[:, 0] = 4.0
    p[:, 3] = np.log((nx - 14.0) / 3.0)   # right end 4 + 3 sigma: inside the last brick but one
    p[:more, 3] = np.log(2.0 * nx)
    og = oracle.Grid(nx, 8, 8)
    off = oracle.brick_lists(p, og, oracle.Config())["gm_off"]
    assert off[min(n, 64)] == 64 * bricks + more
    _check(p, og)


def test_bins_wide_time_follows_the_pairs():
    """64 Gaussians on 16,384 bricks are one tile's work: binning them takes no longer than a few times what as
    many pairs of narrow Gaussians take (2.7 times; 100 times before heavy tiles were shared out; the bound is 6)."""
    import torch
    from paper_2603_09621_gb300 import gs
    grid, cfg = gs.Grid(256, 256, 128), gs.Config()

    def time_of(params):
        n, cap = params.shape[0], 1_200_000
        bins, ws = gs.Bins(n, cap, grid, cfg), gs.Workspace(n, cap, grid, cfg)
        best, pairs = 1e9, 0
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            gs.gs_bin_bricks(params, grid, cfg, bins, ws)
            b.record()
            b.synchronize()
            best, pairs = min(best, a.elapsed_time(b)), bins.npairs()
        return best, pairs

    wide, p_wide = time_of(to_dev(_cover(64, (256, 256, 128))))
    d = inputs.gaussian_cloud(1, 280_000, grid.shape, scale_range=(0.5, 1.5))
    narrow, p_narrow = time_of(to_dev(cloud_params(d)))
    assert p_wide == 64 * 16_384 and 0.8 * p_wide < p_narrow < 1.2 * p_wide
    assert wide < 6 * narrow, (wide, narrow)
