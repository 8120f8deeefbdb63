"""The sort around the number of tiles up to which a pass is one kernel (512 tiles of
4096 positions, one spare per table): the order read back must be the stable one,
with uneven tables, hot rows, and out-of-range lookups."""

import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n", [1, 4096, 4097, 509 * 4096 - 1, 509 * 4096, 510 * 4096 + 5])
@pytest.mark.parametrize("rows", [200, 70_000])
@pytest.mark.parametrize("weighted", [False, True])
def test_order_is_stable(n, rows, weighted):
    from paper_2609_30656_gb300.tbe import TBE
    g = torch.Generator(device=DEV).manual_seed(n + rows)
    # two tables, the second with a twentieth of the lookups (one lookup per bag;
    # a table's missing bags are empty)
    cut = n - n // 20
    batch = cut
    lens = torch.zeros(2 * batch, dtype=torch.int64, device=DEV)
    lens[:cut] = 1
    lens[batch:batch + n - cut] = 1
    off = torch.zeros(2 * batch + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(lens, 0)
    ind = torch.floor(rows * torch.rand(n, generator=g, device=DEV) ** 4).long()
    ind[torch.rand(n, generator=g, device=DEV) < 0.01] = rows + 7
    m = TBE([torch.zeros(rows, 4, device=DEV) for _ in range(2)])
    probe = m.alloc_grad(0, 0, size_only=True)
    w = torch.ones(n, device=DEV) if weighted else None
    m.backward_into(probe, ind, off, torch.zeros(batch, 8, device=DEV), w)
    got = m.sorted_payloads(n)
    m.get_error()
    key = torch.clamp(ind, max=rows) + (torch.arange(n, device=DEV) >= cut) * (rows + 1)
    order = torch.sort(key, stable=True).indices
    if not weighted:
        bags = torch.where(order < cut, order, batch + order - cut)
        order = torch.where(ind[order] < rows, bags, 0xFFFFFFFF)
    assert torch.equal(got, order)
