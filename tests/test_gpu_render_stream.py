"""render() on a stream other than the current one, whose outputs come from the current stream's
allocator pool."""
import pytest

from helpers import cloud_params, to_dev
from paper_2603_09621_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("capacity", [None, 100])
def test_render_on_side_stream_waits_for_the_blocks_last_use(capacity):
    """The outputs' blocks were given up on the current stream while a kernel that writes them is still
    queued there (behind a pause of some milliseconds): the side stream's render comes after it."""
    import torch
    from paper_2603_09621_gb300 import gs
    grid = gs.Grid(96, 80, 64)
    p = to_dev(cloud_params(inputs.gaussian_cloud(3, 3000, grid.shape)))
    I0, W0, _, _ = gs.render(p, grid)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    old = [torch.empty(grid.shape, device="cuda") for _ in range(2)]
    blocks = {t.data_ptr() for t in old}
    torch.cuda._sleep(20_000_000)
    for t in old:
        t.fill_(float("nan"))
    del t, old
    I, W, bins, ws = gs.render(p, grid, capacity=capacity, stream=side)
    torch.cuda.synchronize()
    assert torch.equal(I, I0) and torch.equal(W, W0) and bins.status() == 0
    if not blocks & {I.data_ptr(), W.data_ptr()}:
        pytest.skip("the allocator did not hand the blocks out again")
