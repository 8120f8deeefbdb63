"""Runs of equal row ids against the cells they are cut into (32 sorted positions
in a call this small): runs that end on, before and after cell edges, that cover
whole cells (split, combined by the fix-up, above 32 pieces by a block), and
out-of-range lookups that fill cells of their own. Integer gradients make every
sum exact, so the results equal the oracle's bit for bit."""

import numpy as np
import pytest
import torch

import oracle
from tests.helpers import table_meta

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _problem(counts, dead, dim, seed):
    g = torch.Generator().manual_seed(seed)
    rows = torch.repeat_interleave(torch.arange(len(counts)), torch.tensor(counts))
    rows = torch.cat([rows, torch.full((dead,), len(counts) + 3)])
    ind = torch.cat([rows[torch.randperm(rows.numel(), generator=g)] for _ in range(2)])
    batch = rows.numel()  # two tables, one lookup per bag
    off = torch.arange(2 * batch + 1)
    go = torch.randint(-8, 9, (batch, 2 * dim), generator=g).float()
    tables = [torch.randint(-8, 9, (len(counts), dim), generator=g).float() for _ in range(2)]
    return tables, ind, off, go, batch


@pytest.mark.parametrize("dim", [4, 20, 64, 128, 256])
@pytest.mark.parametrize("counts,dead", [
    ([1, 31, 32, 33, 1, 62, 64, 65, 3], 0),
    ([32] * 7, 64),
    ([33, 63, 95, 96, 97, 1, 1, 1], 5),
    ([1] * 40 + [1100, 31] + [1] * 3 + [2500], 100),
    ([5000], 1),
    ([1], 40),
])
@pytest.mark.parametrize("weighted", [False, True])
def test_runs_around_cell_edges(counts, dead, dim, weighted):
    from paper_2609_30656_gb300.tbe import TBE
    tables, ind, off, go, batch = _problem(counts, dead, dim, len(counts) + dead + dim)
    w = torch.randint(1, 3, (ind.numel(),)).float() if weighted else None
    dw = None if w is None else w.to(DEV)
    keep = ind < len(counts)
    res = oracle.backward(*table_meta(tables), batch, torch.where(keep, ind, 0), off, go,
                          weights=torch.where(keep, torch.ones_like(ind).float() if w is None else w, 0.0), mean=False)
    m = TBE([t.to(DEV) for t in tables])
    g = m.backward(ind.to(DEV), off.to(DEV), go.to(DEV), dw)
    assert m.get_error() == (2 if dead else 0)
    U = g.num_unique
    assert U == res.num_unique
    np.testing.assert_array_equal(g.unique_ids[:U].cpu().numpy(), res.uniq)
    np.testing.assert_array_equal(g.table_offsets.cpu().numpy(), res.table_offsets)
    np.testing.assert_array_equal(g.grad_offsets[:U + 1].cpu().numpy(), res.grad_offsets)
    np.testing.assert_array_equal(g.grads.cpu().double().numpy(), res.grads)
    # the fused step writes what the two-pass step writes
    fused, two = [t.to(DEV).clone() for t in tables], [t.to(DEV).clone() for t in tables]
    TBE(fused).backward_apply(ind.to(DEV), off.to(DEV), go.to(DEV), dw, optimizer="sgd", lr=0.5)
    TBE(two).apply_sparse(g, optimizer="sgd", lr=0.5)
    torch.cuda.synchronize()
    for a, b in zip(fused, two):
        assert torch.equal(a, b)
