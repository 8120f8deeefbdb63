"""A size query finished from its own sorted runs (cb_tbe_backward_finish) gives the
bits of a full backward, and is refused when the workspace holds no such query."""

import ctypes

import pytest
import torch

from tests.helpers import random_problem

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _finish(m, g, ind, off, go, w):
    return m._backward_into(m._lib.cb_tbe_backward_finish, g, ind, off, go, w)


@pytest.mark.parametrize("weighted,pooling", [(False, "sum"), (True, "sum"), (False, "mean")])
@pytest.mark.parametrize("batch,max_len", [(1, 1), (40, 30), (300, 900)])
def test_finish_gives_the_full_calls_bits(weighted, pooling, batch, max_len):
    from paper_2609_30656_gb300.tbe import TBE
    tables, ind, off, w = random_problem(5, dims=(8, 64, 256), rows=(3, 700, 90), batch=batch, max_len=max_len,
                                         weighted=weighted, empty_frac=0.1)
    ind, off = ind.to(DEV), off.to(DEV)
    w = None if w is None else w.to(DEV)
    go = torch.randn(batch, 328, device=DEV)
    m = TBE([t.to(DEV) for t in tables], pooling=pooling, validate=True)
    n = ind.numel()
    full = m.alloc_grad(n, n * 256)
    m.backward_into(full, ind, off, go, w)
    got = m.backward(ind, off, go, w)
    U, F = full.num_unique, full.num_floats
    assert (got.num_unique, got.num_floats) == (U, F)
    assert torch.equal(got.unique_ids[:U], full.unique_ids[:U])
    assert torch.equal(got.grad_offsets[:U + 1], full.grad_offsets[:U + 1])
    assert torch.equal(got.table_offsets, full.table_offsets)
    assert torch.equal(got.grads[:F], full.grads[:F])


def test_finish_needs_the_query_before_it():
    from paper_2609_30656_gb300.tbe import CB_ERR_CAPACITY, TBE, CbTbeError
    tables, ind, off, _ = random_problem(6, batch=30)
    ind, off = ind.to(DEV), off.to(DEV)
    go = torch.randn(30, sum(t.shape[1] for t in tables), device=DEV)
    m = TBE([t.to(DEV) for t in tables])
    n = ind.numel()
    g = m.alloc_grad(n, n * 24)
    probe = m.alloc_grad(0, 0, size_only=True)
    with pytest.raises(CbTbeError):
        _finish(m, g, ind, off, go, None)          # no query yet
    m.backward_into(probe, ind, off, go)
    with pytest.raises(CbTbeError):
        _finish(m, g, ind[:-1], off, go, None)     # another batch
    with pytest.raises(CbTbeError):
        _finish(m, g, ind, off, go, torch.rand(n, device=DEV))  # another kind of payload
    _finish(m, g, ind, off, go, None)
    with pytest.raises(CbTbeError):
        _finish(m, g, ind, off, go, None)          # finished already
    m.backward_into(probe, ind, off, go)
    m.forward(ind, off)
    with pytest.raises(CbTbeError):
        _finish(m, g, ind, off, go, None)          # the forward used the workspace
    m.backward_into(probe, ind, off, go)
    small = m.alloc_grad(1, 8)
    _finish(m, small, ind, off, go, None)
    assert m.get_error() == CB_ERR_CAPACITY
    assert small.num_unique == probe.num_unique


@pytest.mark.parametrize("step", ["backward", "finish", "apply"])
@pytest.mark.parametrize("earlier", [False, True])
def test_nothing_is_summed_in_an_order_that_timed_out(step, earlier):
    """Neither an earlier error of the call (an index out of range) nor one that the host
    read between a query and its finish hides that the sort gave up."""
    from paper_2609_30656_gb300.tbe import CB_DEBUG_FORCE_LOOKBACK_TIMEOUT, CB_ERR_INDEX_OOB, CB_ERR_TIMEOUT, TBE
    tables, ind, off, _ = random_problem(36, rows=(1000, 1000, 1000), batch=400, max_len=60)
    if earlier:
        ind[0] = -1
    ind, off = ind.to(DEV), off.to(DEV)
    go = torch.randn(400, sum(t.shape[1] for t in tables), device=DEV)
    m = TBE([t.to(DEV) for t in tables], extra_flags=CB_DEBUG_FORCE_LOOKBACK_TIMEOUT)
    before = [t.clone() for t in m.tables]
    g = m.alloc_grad(ind.numel(), ind.numel() * 24)
    for x in (g.unique_ids, g.grads):
        x.fill_(-7)
    if step == "apply":
        m.backward_apply(ind, off, go, optimizer="sgd", lr=1.0)
        assert all(torch.equal(a, b) for a, b in zip(before, m.tables))
    elif step == "backward":
        m.backward_into(g, ind, off, go)
    else:
        m.backward_into(m.alloc_grad(0, 0, size_only=True), ind, off, go)
        assert m.get_error() == (CB_ERR_INDEX_OOB if earlier else CB_ERR_TIMEOUT)
        _finish(m, g, ind, off, go, None)
    assert m.get_error() == (CB_ERR_INDEX_OOB if earlier and step != "finish" else CB_ERR_TIMEOUT)
    assert bool((g.unique_ids == -7).all()) and bool((g.grads == -7).all())


@pytest.mark.parametrize("other", ["indices", "offsets", "weights", "stream"])
def test_finish_refuses_another_batch_of_the_same_size(other):
    from paper_2609_30656_gb300.tbe import TBE, CbTbeError
    tables, ind, off, w = random_problem(7, batch=30, weighted=True)
    args = {"indices": ind.to(DEV), "offsets": off.to(DEV), "weights": w.to(DEV)}
    go = torch.randn(30, sum(t.shape[1] for t in tables), device=DEV)
    m = TBE([t.to(DEV) for t in tables])
    want = m.backward(args["indices"], args["offsets"], go, args["weights"])
    g = m.alloc_grad(ind.numel(), ind.numel() * 24)
    g.grads.fill_(-7)
    m.backward_into(m.alloc_grad(0, 0, size_only=True), args["indices"], args["offsets"], go, args["weights"])
    torch.cuda.synchronize()
    mine = dict(args)
    stream = torch.cuda.Stream() if other == "stream" else torch.cuda.current_stream()
    if other != "stream":
        mine[other] = mine[other].clone()
    with pytest.raises(CbTbeError), torch.cuda.stream(stream):
        _finish(m, g, mine["indices"], mine["offsets"], go, mine["weights"])
    torch.cuda.synchronize()
    assert bool((g.grads == -7).all())
    _finish(m, g, args["indices"], args["offsets"], go, args["weights"])  # the query still stands
    assert torch.equal(g.grads[:want.num_floats], want.grads[:want.num_floats])


def test_a_query_that_failed_is_not_finished():
    from paper_2609_30656_gb300.tbe import CB_ERR_INDEX_OOB, CB_ERR_INVALID_ARG, TBE, CbTbeError
    tables, ind, off, _ = random_problem(8, batch=30)
    ind[3] = 1 << 40
    ind, off = ind.to(DEV), off.to(DEV)
    go = torch.randn(30, sum(t.shape[1] for t in tables), device=DEV)
    m = TBE([t.to(DEV) for t in tables], validate=True)
    g = m.alloc_grad(ind.numel(), ind.numel() * 24)
    with pytest.raises(CbTbeError) as e:
        m.backward_into(m.alloc_grad(0, 0, size_only=True), ind, off, go)
    assert e.value.status == CB_ERR_INDEX_OOB
    with pytest.raises(CbTbeError) as e:
        _finish(m, g, ind, off, go, None)
    assert e.value.status == CB_ERR_INVALID_ARG
