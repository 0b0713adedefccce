"""compams_collect through CompAMSOptimizer.collect: a row of G is the concatenation of the parameters' gradients, bit
for bit, whatever the tensors' sizes, the row's 16-byte phase and the gradients' memory layout."""
import pytest
import torch

from paper_2205_05632_b200 import BLOCKSIGN
from paper_2205_05632_b200.optim import CompAMSOptimizer

pytestmark = pytest.mark.gpu

TILE = 4096


@pytest.mark.parametrize("sizes", [
    [1], [2, 1, 3], [TILE - 1, TILE, TILE + 1, 5], [3, 2 * TILE, 1, 3 * TILE + 2], [7] * 160, [5] * 161 + [TILE, 9],
    [2 * TILE + k for k in range(1, 9)],
])
@pytest.mark.parametrize("layout", ["packed", "offset", "transposed", "missing"])
def test_collected_rows_are_the_gradients_bit_for_bit(sizes, layout):
    gen = torch.Generator(device="cuda").manual_seed(len(sizes) + sum(sizes))
    params = [torch.nn.Parameter(torch.zeros(s, device="cuda")) for s in sizes]
    if layout == "transposed":
        params = [torch.nn.Parameter(torch.zeros(2, s, device="cuda")) for s in sizes]
    opt = CompAMSOptimizer(params, 3, BLOCKSIGN)
    opt.G.fill_(float("nan"))
    want = torch.empty_like(opt.G)
    for worker in range(3):
        lo = 0
        for k, p in enumerate(params):
            g = torch.randn(p.numel() + 1, generator=gen, device="cuda")
            g = g[1:] if layout == "offset" else g[:-1]  # 4 bytes past an allocation's start, or at it
            g = g.view(-1, 2).t() if layout == "transposed" else g
            p.grad = None if layout == "missing" and (k + worker) % 2 == 0 else g
            want[worker, lo:lo + p.numel()] = 0.0 if p.grad is None else g.reshape(-1)
            lo += p.numel()
        opt.collect(worker)
        assert all(p.grad is None for p in params)
    assert torch.equal(opt.G.view(torch.int32), want.view(torch.int32))
    opt.close()


@pytest.mark.parametrize("sizes", [[0, 3], [5, 0], [0, 0, TILE + 1, 0, 2, 0], [7] * 80 + [0] + [7] * 80])
def test_parameters_without_elements_are_passed_over(sizes):
    # with the whole vector as one block they are no block of their own
    params = [torch.nn.Parameter(torch.zeros(s, device="cuda")) for s in sizes]
    opt = CompAMSOptimizer(params, 2, BLOCKSIGN, whole_vector=True)
    opt.G.fill_(float("nan"))
    want = torch.arange(2 * sum(sizes), device="cuda").float().view(2, -1)
    for worker in range(2):
        for p, g in zip(params, torch.split(want[worker], sizes)):
            p.grad = g.clone()
        opt.collect(worker)
        assert all(p.grad is None for p in params)
    assert torch.equal(opt.G, want)
    opt.step()
    opt.close()
