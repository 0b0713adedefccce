"""compams_collect through CompAMSOptimizer.collect: a row of G is the concatenation of the parameters' gradients, bit
for bit, whatever the tensors' sizes, the row's 16-byte phase and the gradients' memory layout."""
import pytest
import torch

from paper_2205_05632_b200 import BLOCKSIGN, CompAMSError
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


def test_gradients_that_are_not_packed_float32_on_the_device_are_made_so():
    # what the copy of one tensor after the other took: other types and devices, lazily negated values
    params = [torch.nn.Parameter(torch.zeros(s, device="cuda")) for s in ([70], [1], [8, 9], [33])]
    opt = CompAMSOptimizer(params, 1, BLOCKSIGN)
    gen = torch.Generator(device="cuda").manual_seed(3)
    for change in (lambda t: t.half(), lambda t: t.bfloat16(), lambda t: t.double(), lambda t: t.cpu()):
        for p in params:
            p.data = change(p.data)
            p.grad = torch.randn(p.shape, generator=gen, device="cuda").to(p.device, p.dtype)
        want = torch.cat([p.grad.reshape(-1).float().cuda() for p in params])
        opt.collect(0)
        assert torch.equal(opt.G[0], want)
    for p in params:
        p.data = torch.zeros(p.shape, device="cuda")
        z = torch.view_as_complex(torch.randn(*p.shape, 2, generator=gen, device="cuda"))
        p.grad = z.conj().imag
        assert p.grad.is_neg()
    want = torch.cat([p.grad.reshape(-1) for p in params]).resolve_neg()
    opt.collect(0)
    assert torch.equal(opt.G[0], want)
    params[2].data = torch.zeros(5, device="cuda")
    params[2].grad = torch.ones(5, device="cuda")
    with pytest.raises(CompAMSError):
        opt.collect(0)
    opt.close()
