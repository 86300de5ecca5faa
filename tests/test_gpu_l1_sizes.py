"""gs_l1_loss where its loop over a fixed grid of 524,288 values can go wrong: whole and partial strides, one and
two in flight, remainders of a quad; gradient exact, loss the same bits with and without alignment and gradient."""
import pytest

pytestmark = pytest.mark.gpu

STRIDE = 4 * 1024 * 128


@pytest.mark.parametrize("n", [1, 3, 4, 5, 511, STRIDE - 1, STRIDE, STRIDE + 1, STRIDE + 6,
                               2 * STRIDE - 3, 2 * STRIDE, 2 * STRIDE + 4, 3 * STRIDE - 1, 3 * STRIDE + 2, 5 * STRIDE + 7])
def test_l1_sizes(n):
    import torch
    from paper_2603_09621_gb300 import gs
    ws = gs.Workspace(10, 1000, gs.Grid(8, 8, 8), gs.Config())
    gen = torch.Generator(device="cuda").manual_seed(n)
    pred, target = (torch.randn(n + 1, generator=gen, device="cuda") for _ in range(2))
    target[:n // 3] = pred[:n // 3]      # exact zeros
    got = []
    for off in (0, 1):
        a, t = pred[:n].clone(), target[:n].clone()
        if off:
            a, t = (torch.cat([x[:1], x])[1:] for x in (a, t))
        grad = torch.full((n + 1,), -7.0, device="cuda")
        loss = gs.gs_l1_loss(a, t, ws, dpred=grad[:n])
        inv = 1.0 / torch.tensor(float(n), dtype=torch.float32).item()
        want = torch.sign(a - t) * torch.tensor(inv, dtype=torch.float32, device="cuda")
        assert torch.equal(grad[:n], want) and grad[n] == -7.0
        got += [loss.item(), gs.gs_l1_loss(a, t, ws).item()]
        assert torch.equal(a, pred[:n]) and torch.equal(t, target[:n])
    assert len(set(got)) == 1
    ref = (pred[:n].double() - target[:n].double()).abs().mean().item()
    # a thread adds up to 22 values, then 17 levels of a tree: (22 + 17 + 2) 2^-24 of a sum of magnitudes
    assert abs(got[0] - ref) <= 41 * 2.0**-24 * ref
