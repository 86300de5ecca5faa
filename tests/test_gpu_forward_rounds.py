"""Forward render where its list handling can go wrong: brick lists at the edges of a staging
round (20 records per 4^3 footprint: 40, 80 or 160) and of the four hits an iteration takes, at
every footprint layout of a brick, against the FP64 oracle."""
import functools

import numpy as np
import pytest

from helpers import cloud_params
from paper_2603_09621_gb300 import inputs
from test_gpu_render import check_forward, gpu_render, oracle_ref

pytestmark = pytest.mark.gpu

# partial bricks along every axis; few bricks (a warp per footprint) and many (a quarter-warp)
SHAPES = ((10, 11, 13), (1290, 11, 13))


@functools.lru_cache(maxsize=None)
def _ref(n, shape):
    """n Gaussians whose boxes meet every brick of the grid's first 8^3 voxels, and the oracle on the
    first 24 slices (none reaches further)."""
    import oracle
    d = inputs.gaussian_cloud(n, n, SHAPES[0], scale_range=(1.0, 2.0))
    d["mu"] = (4.0 + 2.0 * (d["mu"] / np.array(SHAPES[0][::-1], np.float32) - 0.5)).astype(np.float32)
    og = oracle.Grid(shape[2], shape[1], min(shape[0], 24))
    params = cloud_params(d)
    return params, og, oracle_ref(params, og)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("brick", [(8, 8, 8), (8, 8, 4), (4, 4, 4), (16, 4, 8), (4, 8, 8), (4, 4, 16)])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 40, 41, 80, 81, 159, 160, 161, 325])
def test_forward_round_edges(n, brick, shape):
    import oracle
    params, og, ref = _ref(n, shape)
    full = oracle.Grid(shape[2], shape[1], shape[0])
    out = gpu_render(params, full, brick=brick, stats=True)
    check_forward(out["I"][:og.nz], out["W"][:og.nz], ref)
    assert not out["W"][og.nz:].any()
    n_eff, n_eval = out["stats"]
    assert abs(int(n_eff) - int(ref["npair"].sum())) <= int(ref["amb"].sum())
    assert n_eval >= n_eff
