"""Bags that span many chunks, at the edges of the fix-up's ways to add their pieces: one
warp up to 32 pieces, a block above, and groups of 128 chunks whose sums are added by the
last block to finish. Whole numbers make every sum exact in fp32, so results are equal."""

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
    added by the whole GPU (about 1.2 times as long; 25 times with one warp per bag)."""
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
