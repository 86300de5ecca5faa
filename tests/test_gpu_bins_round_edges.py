"""Brick lists at the edges of the radix passes' rounds: first-pass tiles of exactly 2,048 pairs (the most that take
rounds of 2,048), 2,304 and 4,608 (one and two rounds of 2,304) and one pair more or fewer, for tiles of 64 and of 256
Gaussians, and later-pass tiles of 2,048. The tile's pairs are asserted, so the cases stay at the edges."""
import numpy as np
import pytest

from test_gpu_bins_tiles import _check

pytestmark = pytest.mark.gpu


def _row(n, bricks, total, tile, extra):
    """n Gaussians on a row of `total` bricks of 8^3, each meeting the first `bricks`; `extra` of the first tile
    meet one more (fewer where negative)."""
    nx = 8 * total
    p = np.zeros((n, 12), np.float32)
    p[:, :3] = (4.0, 4.0, 4.0)
    p[:, 3:6] = np.log(50.0)
    p[:, 6], p[:, 10:] = 1.0, 0.5
    ends = np.full(n, bricks)
    ends[:abs(extra)] += np.sign(extra)
    p[:, 3] = np.log((8.0 * ends - 8.0) / 3.0)   # right end 4 + 3 sigma: the middle of the last brick
    return p, nx


@pytest.mark.parametrize("extra", [-1, 0, 1])
@pytest.mark.parametrize("n,tile,bricks", [(64, 64, 32), (200, 64, 32), (200, 64, 36), (130, 64, 72),
                                           (38_913, 256, 8), (39_100, 256, 9), (38_914, 256, 18)])
@pytest.mark.parametrize("total", [80, 600])
def test_first_pass_round_edges(n, tile, bricks, extra, total):
    import oracle
    p, nx = _row(n, bricks, total, tile, extra)
    og = oracle.Grid(nx, 8, 8)
    off = oracle.brick_lists(p, og, oracle.Config())["gm_off"]
    assert off[tile] == tile * bricks + extra and off[n] == n * bricks + extra
    _check(p, og)


@pytest.mark.parametrize("extra", [-1, 0, 1])
@pytest.mark.parametrize("n", [32, 64, 128])
def test_later_pass_tile_edges(n, extra):
    """2,048, 4,096 and 8,192 pairs and one more or fewer in all, on 600 bricks (two passes)."""
    import oracle
    p, nx = _row(n, 64, 600, 64, extra)
    og = oracle.Grid(nx, 8, 8)
    assert oracle.brick_lists(p, og, oracle.Config())["pair_gid"].size == 64 * n + extra
    _check(p, og)
