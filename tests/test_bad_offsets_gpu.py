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


def _padded_tables(tables):
    bufs = []
    for x in tables:
        buf, y = _padded(x.reshape(-1), MARK)
        bufs.append((buf, y.view(x.shape)))
    return bufs


def _marks_stand(bufs):
    return all(bool((b[:PAD] == MARK).all()) and bool((b[-PAD:] == MARK).all()) for b, _ in bufs)


@pytest.mark.parametrize("seed", [1, 2, 3])
@pytest.mark.parametrize("dims,B,max_len", SHAPES)
def test_backward_sorts_every_lookup_once(dims, B, max_len, seed):
    """Whatever table 1's offsets, the sort's payloads are its lookups, each once, and the
    other tables' gradients and steps are those of the well-formed batch."""
    from paper_2609_30656_gb300.tbe import CB_ERR_INDEX_OOB, TBE
    tables, ind, off, w = random_problem(seed, dims=dims, rows=(70, 500, 300), batch=B, max_len=max_len, weighted=True)
    n = ind.numel()
    bad = _decreasing_inside(off, B, 1, seed + 10).to(DEV)
    _, ind = _padded(ind, -7)
    off, w = off.to(DEV), w.to(DEV)
    go = torch.randn(B, sum(dims), device=DEV)
    bufs = _padded_tables(tables)
    state = [_padded(torch.zeros(t.shape[0]), MARK) for t in tables]
    m = TBE([t for _, t in bufs])
    want = m.backward(ind, off, go, w)
    room = (want.unique_ids.numel() + PAD, want.grads.numel() + PAD)
    g = m.alloc_grad(*room)
    for x in (g.unique_ids, g.grad_offsets, g.grads):
        x.fill_(-7)
    m.backward_into(g, ind, bad, go, w)
    assert m.get_error() != CB_ERR_INDEX_OOB
    assert torch.equal(m.sorted_payloads(n).sort().values, torch.arange(n, device=DEV))
    # as many rows as the well-formed batch touches (they are the same lookups), and nothing past them
    U, F = want.num_unique, want.num_floats
    assert (g.num_unique, g.num_floats) == (U, F)
    assert torch.equal(g.unique_ids[:U], want.unique_ids) and bool((g.unique_ids[U:] == -7).all())
    assert torch.equal(g.grad_offsets[:U + 1], want.grad_offsets) and bool((g.grads[F:] == -7).all())
    f0, f1 = (int(want.grad_offsets[int(want.table_offsets[t])]) for t in (1, 2))
    assert torch.equal(g.grads[:f0], want.grads[:f0]) and torch.equal(g.grads[f1:F], want.grads[f1:F])
    m.backward_apply(ind, bad, go, w, optimizer="adagrad", state=[s for _, s in state])
    assert _marks_stand(bufs) and _marks_stand(state)
