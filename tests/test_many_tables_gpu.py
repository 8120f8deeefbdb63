"""The chunk plan around the number of tables that a block scans in shared memory
(1024): integer tables, so forward and backward equal the oracle's bit for bit."""

import numpy as np
import pytest
import torch

import oracle
from tests.helpers import forward_reference, random_problem, table_meta

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("num_tables", [1, 255, 256, 257, 1023, 1024, 1025, 2100])
def test_forward_and_backward(num_tables):
    from paper_2609_30656_gb300.tbe import TBE
    dims = [4 * (1 + t % 3) for t in range(num_tables)]
    tables, ind, off, _ = random_problem(num_tables, dims=dims, rows=[5] * num_tables, batch=3, max_len=9,
                                         int_valued=True, empty_frac=0.4)
    go = torch.randint(-8, 9, (3, sum(dims))).float()
    m = TBE([t.to(DEV) for t in tables], validate=True)
    y = m.forward(ind.to(DEV), off.to(DEV))
    ref, _ = forward_reference(tables, 3, ind, off, None, False)
    np.testing.assert_array_equal(y.cpu().double().numpy(), ref)
    g = m.backward(ind.to(DEV), off.to(DEV), go.to(DEV))
    res = oracle.backward(*table_meta(tables), 3, ind, off, go, weights=None, mean=False)
    assert g.num_unique == res.num_unique
    np.testing.assert_array_equal(g.unique_ids.cpu().numpy(), res.uniq)
    np.testing.assert_array_equal(g.table_offsets.cpu().numpy(), res.table_offsets)
    np.testing.assert_array_equal(g.grads.cpu().double().numpy(), res.grads)


@pytest.mark.parametrize("num_tables,longest", [(304, 160_000), (305, 31_000), (305, 33_000), (305, 160_000),
                                                (305, 270_000), (1500, 100_000)])
def test_one_long_table_among_many(num_tables, longest):
    """Runs are scanned by small blocks where there are many tables of few cells (32 lookups
    each); one table here has many rounds of such a block."""
    from paper_2609_30656_gb300.tbe import TBE
    g = torch.Generator(device=DEV).manual_seed(longest)
    rows, D, B, long = 1000, 4, 4, num_tables // 2
    lens = torch.randint(0, 3, (num_tables * B,), generator=g, device=DEV)
    lens[long * B:(long + 1) * B] = longest // B
    off = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), lens.cumsum(0)])
    n = int(off[-1])
    ind = torch.randint(0, rows, (n,), generator=g, device=DEV)
    go = torch.randint(-8, 9, (B, num_tables * D), generator=g, device=DEV).float()
    m = TBE([torch.zeros(rows, D, device=DEV) for _ in range(num_tables)], validate=True)
    got = m.backward(ind, off, go)
    bag = torch.repeat_interleave(torch.arange(num_tables * B, device=DEV), lens)
    ids, inverse = torch.unique(bag // B * rows + ind, return_inverse=True)
    want = torch.zeros(ids.numel(), D, dtype=torch.float64, device=DEV)
    cols = go.view(B, num_tables, D).transpose(0, 1).reshape(num_tables * B, D)
    want.index_add_(0, inverse, cols[bag].double())
    assert torch.equal(got.unique_ids, ids)
    assert torch.equal(got.grads.view(-1, D).double(), want)
