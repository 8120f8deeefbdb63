"""Malformed offsets stay inside the caller's buffers and inside their own table.

The lookups stand inside a larger buffer whose other words hold an index that no table
has. So a call that reads a lookup outside [0, n) reports CB_ERR_INDEX_OOB, and one that
writes beside its output leaves a mark in the words around it.
"""

import pytest
import torch

from tests.helpers import random_problem

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
PAD = 1 << 16
MARK = -77.0
# tables of one row layout and of several; batches of one chunk per table and of many
SHAPES = [((16, 16, 16), 40, 30), ((8, 64, 128), 600, 40), ((8, 64, 128), 2000, 60)]


def _padded(x, fill):
    buf = torch.full((x.numel() + 2 * PAD,), fill, dtype=x.dtype, device=DEV)
    buf[PAD:PAD + x.numel()] = x.to(DEV)
    return buf, buf[PAD:PAD + x.numel()]


def _decreasing_inside(off, B, t, seed):
    """off with a few of table t's inner offsets replaced by any others, below 0 and above n too."""
    g = torch.Generator().manual_seed(seed)
    n = int(off[-1])
    off = off.clone()
    at = t * B + 1 + torch.randint(0, B - 1, (max(2, B // 16),), generator=g)
    off[at] = torch.randint(-PAD // 2, n + PAD // 2, at.shape, generator=g)
    assert bool((off[1:] < off[:-1]).any())
    return off


@pytest.mark.parametrize("seed", [1, 2, 3])
@pytest.mark.parametrize("one_type", [True, False])
@pytest.mark.parametrize("dims,B,max_len", SHAPES)
def test_offsets_that_decrease_inside_a_table(dims, B, max_len, one_type, seed):
    from paper_2609_30656_gb300.tbe import CB_ERR_INDEX_OOB, TBE
    tables, ind, off, _ = random_problem(seed, dims=dims, rows=(70, 500, 300), batch=B, max_len=max_len)
    if not one_type:
        tables[2] = tables[2].half()
    bad = _decreasing_inside(off, B, 1, seed).to(DEV)
    _, ind = _padded(ind, -7)
    off = off.to(DEV)
    m = TBE([t.to(DEV) for t in tables])
    want = m.forward(ind, off)
    got = m.forward(ind, bad)
    assert m.get_error() != CB_ERR_INDEX_OOB
    for lo, hi in ((0, dims[0]), (dims[0] + dims[1], sum(dims))):  # the other tables
        assert torch.equal(got[:, lo:hi], want[:, lo:hi])
    go = torch.randn(B, sum(dims), device=DEV)
    buf, gw = _padded(torch.empty(ind.numel()), MARK)
    m.weight_grad(ind, bad, go, out=gw)
    assert m.get_error() != CB_ERR_INDEX_OOB
    assert bool((buf[:PAD] == MARK).all()) and bool((buf[-PAD:] == MARK).all())
    want = m.weight_grad(ind, off, go)
    a, b = int(off[B]), int(off[2 * B])
    assert torch.equal(gw[:a], want[:a]) and torch.equal(gw[b:], want[b:])
