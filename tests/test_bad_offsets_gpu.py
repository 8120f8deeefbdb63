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


# First offsets of the tables as parts of n, and the ranges that the call gives them
# (no range begins before an earlier one's); inner offsets between each pair.
BOUNDARIES = [
    ((0.0, 1.0, 0.0, 1.0), (0.0, 1.0, 1.0, 1.0)),
    ((0.0, 0.1, 0.05, 0.2), (0.0, 0.1, 0.1, 0.2)),
    ((0.0, 0.5, -3.0, 0.6), (0.0, 0.5, 0.5, 0.6)),
    ((0.0, 2.0, 0.2, 0.0), (0.0, 1.0, 1.0, 1.0)),
]


# n around the edges of the chunk lengths (32, 64, .., 512) and of the few-tile sort
@pytest.mark.parametrize("n,copies", [(50, 1), (5000, 1), (640_000, 1), (2_200_000, 1), (10_500_000, 1),
                                      (50, 400), (5000, 400), (640_000, 400)])
@pytest.mark.parametrize("parts,used", BOUNDARIES)
def test_tables_that_begin_before_an_earlier_one(parts, used, copies, n):
    """Three tables, or three and 1197 that begin as the third does (more than one block plans)."""
    from paper_2609_30656_gb300.tbe import CB_ERR_BAD_OFFSETS, SparseGrad, TBE
    rows, D, B = 1000, 4, 16
    T = 3 * copies
    gen = torch.Generator(device=DEV).manual_seed(n)
    _, ind = _padded(torch.randint(0, rows, (n,), generator=gen, device=DEV), -7)
    starts = [int(p * n) for p in parts]
    starts = starts[:3] + [starts[2]] * (T - 3) + starts[3:]
    off = torch.cat([torch.linspace(a, b, B + 1, dtype=torch.float64, device=DEV)[:B].long()
                     for a, b in zip(starts, starts[1:])] + [torch.tensor(starts[-1:], device=DEV)])
    held = [int(p * n) for p in used]
    held = held[:3] + [held[2]] * (T - 3) + held[3:]
    w = torch.rand(n, generator=gen, device=DEV)
    go = torch.randn(B, T * D, generator=gen, device=DEV)
    bufs = _padded_tables([torch.randn(rows, D) for _ in range(T)])
    tables = [t for _, t in bufs]
    m = TBE(tables)
    ids = torch.cat([ind[a:b].unique() + t * rows for t, (a, b) in enumerate(zip(held, held[1:]))])
    U = ids.numel()
    (bi, unique_ids), (bo, grad_offsets), (bg, grads) = (_padded(torch.zeros(k, dtype=d), -7) for k, d in (
        (U, torch.int64), (U + 1, torch.int64), (U * D, torch.float32)))
    sizes = torch.zeros(2, dtype=torch.int64, device=DEV)
    g = SparseGrad(unique_ids, torch.zeros(T + 1, dtype=torch.int64, device=DEV), grad_offsets, grads, sizes[:1], sizes[1:])
    m.backward_into(g, ind, off, go, w)
    assert m.get_error() == CB_ERR_BAD_OFFSETS
    assert torch.equal(m.sorted_payloads(n)[:held[-1]].sort().values, torch.arange(held[-1], device=DEV))
    assert (g.num_unique, g.num_floats) == (U, U * D)
    assert torch.equal(unique_ids, ids) and torch.equal(grad_offsets, torch.arange(U + 1, device=DEV) * D)
    for b in (bi, bo, bg):
        assert bool((b[:PAD] == -7).all()) and bool((b[-PAD:] == -7).all())
    m.backward_apply(ind, off, go, w, optimizer="sgd", lr=0.5)
    assert m.get_error() == CB_ERR_BAD_OFFSETS and _marks_stand(bufs)
    buf, gw = _padded(torch.empty(n), MARK)
    m.weight_grad(ind, off, go, out=gw)
    assert m.get_error() == CB_ERR_BAD_OFFSETS
    assert bool((buf[:PAD] == MARK).all()) and bool((buf[-PAD:] == MARK).all())
    m.forward(ind, off, w)
    assert m.get_error() == CB_ERR_BAD_OFFSETS
    # the handle is as good as new
    good = (torch.arange(T * B + 1, device=DEV) * n) // (T * B)
    other = TBE(tables)
    assert torch.equal(m.forward(ind, good, w), other.forward(ind, good, w))
    x, y = m.backward(ind, good, go, w), other.backward(ind, good, go, w)
    assert torch.equal(x.unique_ids, y.unique_ids) and torch.equal(x.grads, y.grads) and m.get_error() == 0
