"""A call's kernels overlap each other's launches (programmatic stream serialization):
captured into a CUDA graph and replayed, and enqueued back to back on two streams,
they give the bits of calls that the host waits for one by one."""

import pytest
import torch

from tests.helpers import random_problem

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _batches(count, batch=64, max_len=60):
    out = []
    for k in range(count):
        tables, ind, off, w = random_problem(50 + k, dims=(64, 8, 256), rows=(900, 40, 3000), batch=batch,
                                             max_len=max_len, weighted=True)
        out.append((ind, off, w, torch.randn(batch, 328)))
    return tables, out


def _calls(m, g, ind, off, w, go):
    y = m.forward(ind, off, w)
    m.backward_into(g, ind, off, go, w)
    return [y, m.weight_grad(ind, off, go), g.num_unique_dev.clone(), g.num_floats_dev.clone(), g.unique_ids.clone(),
            g.grads.clone()]


def _zeroed(m, n):
    g = m.alloc_grad(n, n * 256)
    for t in (g.unique_ids, g.grad_offsets, g.grads):
        t.zero_()
    return g


def test_replayed_graph():
    from paper_2609_30656_gb300.tbe import TBE
    tables, batches = _batches(3)
    n = min(b[0].numel() for b in batches)
    m = TBE([t.to(DEV) for t in tables])
    m.reserve(64, n)
    # one number of lookups for every batch: the last bag of each is cut
    fixed = [(i[:n].to(DEV), o.clamp(max=n).to(DEV), w[:n].to(DEV), go.to(DEV)) for i, o, w, go in batches]
    want = []
    for b in fixed:
        want.append([t.clone() for t in _calls(m, _zeroed(m, n), *b)])
        torch.cuda.synchronize()
    static = [t.clone() for t in fixed[0]]
    g = _zeroed(m, n)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = _calls(m, g, *static)
    for b, ref in zip(fixed, want):
        for s, t in zip(static, b):
            s.copy_(t)
        for t in (g.unique_ids, g.grad_offsets, g.grads):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for a, r in zip(got, ref):
            assert torch.equal(a, r)


def test_two_streams_back_to_back():
    from paper_2609_30656_gb300.tbe import TBE
    tables, batches = _batches(2, batch=200, max_len=100)
    dev = [tuple(t.to(DEV) for t in b) for b in batches]
    handles = [TBE([t.to(DEV) for t in tables]) for _ in dev]
    want = []
    for m, b in zip(handles, dev):
        want.append(_calls(m, _zeroed(m, b[0].numel()), *b))
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in dev]
    grads = [_zeroed(m, b[0].numel()) for m, b in zip(handles, dev)]
    torch.cuda.synchronize()
    for _ in range(5):
        got = []
        for m, b, g, s in zip(handles, dev, grads, streams):
            with torch.cuda.stream(s):
                got.append(_calls(m, g, *b))
        torch.cuda.synchronize()
        for a, r in zip(got, want):
            for x, z in zip(a, r):
                assert torch.equal(x, z)
