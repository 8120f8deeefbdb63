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
