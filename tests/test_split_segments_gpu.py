"""Bags, and runs of one row's lookups, that span many chunks, at the edges of the fix-up's
ways to add their pieces: one warp up to 32 pieces, a block up to 256, and above that groups
of 128 chunks whose sums are added by the last block to finish. Whole numbers make every sum exact in
fp32, so results are equal."""

import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
C = 32  # lookups per chunk in calls of up to 600 thousand lookups


def _times(call, repeats=7):
    call()
    took = []
    for _ in range(repeats):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        took.append(a.elapsed_time(b))
    return sorted(took)[repeats // 2]


# bag lengths in lookups, in a table: pieces around 32, group edges, several heavy bags in a row
LENGTHS = [
    [5, 4 * C + 1, 32 * C, 33 * C, 34 * C + 7, 3],
    [126 * C, 127 * C + 1, 128 * C, 129 * C - 1],
    [0, 1, 255 * C + 31, 0, 257 * C, 2],
    [40 * C + 3] * 9,
    [9 * C, 4000 * C + 17, 0, 5],
]


@pytest.mark.parametrize("lengths", LENGTHS)
@pytest.mark.parametrize("dim,dtype,out", [(4, torch.float32, torch.float32), (12, torch.float32, torch.float32),
                                           (64, torch.float32, torch.float32), (200, torch.float16, torch.float32),
                                           (384, torch.bfloat16, torch.float32), (512, torch.float16, torch.float32),
                                           (64, torch.float16, torch.bfloat16)])
def test_bags_of_many_pieces(lengths, dim, dtype, out):
    from paper_2609_30656_gb300.tbe import TBE
    g = torch.Generator(device=DEV).manual_seed(dim)
    B, T, rows = len(lengths), 3, 50
    # the second table's heavy bags begin elsewhere within their groups
    lens = torch.tensor(lengths + [7] * B + lengths, device=DEV)
    off = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), lens.cumsum(0)])
    n = int(off[-1])
    ind = torch.randint(0, rows, (n,), generator=g, device=DEV)
    tables = [torch.randint(-8, 9, (rows, dim), generator=g, device=DEV).to(dtype) for _ in range(T)]
    want = torch.zeros(T * B, dim, dtype=torch.float64, device=DEV)
    bag = torch.repeat_interleave(torch.arange(T * B, device=DEV), lens)
    for t in range(T):
        a, b = int(off[t * B]), int(off[(t + 1) * B])
        want.index_add_(0, bag[a:b], tables[t][ind[a:b]].double())
    want = want.view(T, B, dim)
    got = TBE(tables, out_dtype=out).forward(ind, off)
    assert torch.equal(got, want.transpose(0, 1).reshape(B, T * dim).to(out))
    mean = TBE(tables, pooling="mean", out_dtype=out).forward(ind, off)
    want = want / lens.view(T, B, 1).clamp(min=1)
    eps = 2 ** -8 if out == torch.bfloat16 else 2 ** -23  # one rounding of the quotient, of one in fp64 or fp32
    assert torch.allclose(mean.double(), want.transpose(0, 1).reshape(B, T * dim), rtol=2 * eps, atol=0)


def test_one_bag_takes_no_longer_than_many():
    """A million lookups in one bag against the same in bags of a thousand: the pieces are
    added by the whole GPU (a little longer; 25 times as long with one warp per bag)."""
    from paper_2609_30656_gb300.tbe import TBE
    n, rows = 1_000_000, 100_000
    ind = torch.randint(0, rows, (n,), device=DEV)
    m = TBE([torch.randn(rows, 64, device=DEV)])
    took = []
    for B in (1, 1000):
        off = torch.arange(B + 1, device=DEV) * (n // B)
        out = torch.empty(B, 64, device=DEV)
        took.append(_times(lambda: m.forward(ind, off, out=out)))
    assert took[0] < 4 * took[1], took


@pytest.mark.parametrize("lengths", LENGTHS)
@pytest.mark.parametrize("invalid", [False, True])
@pytest.mark.parametrize("dim,out", [(4, torch.float32), (64, torch.float32), (200, torch.float32),
                                     (384, torch.bfloat16), (512, torch.float16)])
def test_runs_of_many_pieces(lengths, invalid, dim, out):
    """Row r of every table is looked up lengths[r] times, the last row (or, invalid: no
    row, a run that is dropped) as often as a few chunks hold."""
    from paper_2609_30656_gb300.tbe import CB_ERR_INDEX_OOB, TBE
    g = torch.Generator(device=DEV).manual_seed(dim)
    T, B, rows = 3, 40, len(lengths) + 1
    counts = [lengths + [0], [7] * (rows - 1) + [150 * C], lengths + [131 * C + 2]]
    if invalid:  # index `rows` is out of range
        counts = [c[:-1] + [0, c[-1]] for c in counts]
    ind = torch.cat([torch.repeat_interleave(torch.arange(len(c), device=DEV), torch.tensor(c, device=DEV))[
        torch.randperm(sum(c), generator=g, device=DEV)] for c in counts])
    starts = [0]
    for c in counts:
        starts.append(starts[-1] + sum(c))
    off = torch.cat([(a + (torch.arange(B, device=DEV) * (b - a)) // B) for a, b in zip(starts, starts[1:])]
                    + [torch.tensor(starts[-1:], device=DEV)])
    go = torch.randint(-8, 9, (B, T * dim), generator=g, device=DEV).to(out)
    tables = [torch.randint(-8, 9, (rows, dim), generator=g, device=DEV).float() for _ in range(T)]
    bag = torch.repeat_interleave(torch.arange(T * B, device=DEV), off[1:] - off[:-1])
    ids, want = [], []
    for t in range(T):
        a, b = starts[t], starts[t + 1]
        G = torch.zeros(rows + 1, dim, dtype=torch.float64, device=DEV)
        G.index_add_(0, ind[a:b], go[bag[a:b] - t * B, t * dim:(t + 1) * dim].double())
        seen = ind[a:b].unique()
        seen = seen[seen < rows]
        ids.append(seen + t * rows)
        want.append(G[:rows])
    m = TBE(tables, out_dtype=out)
    got = m.backward(ind, off, go)
    assert (m.get_error() == CB_ERR_INDEX_OOB) == invalid
    assert torch.equal(got.unique_ids, torch.cat(ids))
    expect = torch.cat([w[i - t * rows] for t, (w, i) in enumerate(zip(want, ids))])
    assert torch.equal(got.grads.view(-1, dim).double(), expect)
    assert torch.equal(m.backward(ind, off, go).grads, got.grads)
    before = [t.clone() for t in m.tables]
    m.backward_apply(ind, off, go, optimizer="sgd", lr=0.25)
    for t, w, x in zip(m.tables, want, before):
        assert torch.equal(t.double(), x.double() - 0.25 * w)


def test_one_hot_row_takes_no_longer_than_many():
    """A million lookups of one row against the same over the table."""
    from paper_2609_30656_gb300.tbe import TBE
    n, rows, B = 1_000_000, 100_000, 1000
    m = TBE([torch.randn(rows, 64, device=DEV)])
    off = torch.arange(B + 1, device=DEV) * (n // B)
    go = torch.randn(B, 64, device=DEV)
    g = m.alloc_grad(rows, rows * 64)
    took = []
    for ind in (torch.full((n,), 7, device=DEV), torch.randint(0, rows, (n,), device=DEV)):
        took.append(_times(lambda: m.backward_into(g, ind, off, go)))
    assert took[0] < 2 * took[1], took
