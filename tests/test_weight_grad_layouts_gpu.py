"""The weight gradient on every layout of a row over a warp, around the number of
lookups a lane group takes at a time (8, 32 per batch), against the oracle; and
out-of-range lookups, and rows with infinities, next to ordinary ones."""

import numpy as np
import pytest
import torch

import oracle
from tests.helpers import inject_out_of_range

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
LENGTHS = [1, 0, 7, 8, 9, 15, 16, 17, 31, 0, 0, 32, 33, 1, 1, 1, 63, 64, 65, 2, 200, 0]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16])
@pytest.mark.parametrize("mean", [False, True])
@pytest.mark.parametrize("bad", [0.0, 0.3])
def test_layouts(dtype, mean, bad):
    from paper_2609_30656_gb300.tbe import TBE
    per = 4 if dtype == torch.float32 else 8
    g = torch.Generator().manual_seed(3)
    dims = [min(v * per, 512) for v in (1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 64, 65, 128)]
    tables = [torch.randn(50, d, generator=g).to(dtype) for d in dims]
    batch = len(LENGTHS)
    off = torch.zeros(len(dims) * batch + 1, dtype=torch.int64)
    off[1:] = torch.cumsum(torch.tensor(LENGTHS * len(dims)), 0)
    ind = torch.randint(0, 50, (int(off[-1]),), generator=g)
    go = torch.randn(batch, sum(dims), generator=g)
    drop = torch.zeros(ind.numel(), dtype=torch.bool)
    sent = ind
    if bad:
        sent, drop = inject_out_of_range(tables, ind, off, batch, 4, frac=bad)
    m = TBE([t.to(DEV) for t in tables], pooling="mean" if mean else "sum")
    got = m.weight_grad(sent.to(DEV), off.to(DEV), go.to(DEV)).cpu().double().numpy()
    assert m.get_error() == (2 if bad else 0)
    ref = oracle.weight_grad(tables, batch, ind, off, go, mean=mean)
    scale = oracle.weight_grad([t.abs() for t in tables], batch, ind, off, go.abs(), mean=mean)
    keep = ~drop.numpy()
    assert (got[~keep] == 0).all()
    # a dot product of up to 512 fp32 terms: the 1e-5 of the other weight-gradient tests
    assert (np.abs(got - ref)[keep] <= 1e-5 * scale[keep] + 1e-30).all()


def test_infinities_stay_with_their_lookup():
    from paper_2609_30656_gb300.tbe import TBE
    table = torch.ones(4, 12)  # 3 vectors on 4 lanes: one lane past the row
    table[1, 0] = float("inf")
    off = torch.tensor([0, 40])
    ind = torch.arange(40) % 4
    got = TBE([table.to(DEV)]).weight_grad(ind.to(DEV), off.to(DEV), torch.ones(1, 12, device=DEV)).cpu()
    want = torch.where(ind == 1, torch.tensor(float("inf")), torch.tensor(12.0))
    assert torch.equal(got, want)
