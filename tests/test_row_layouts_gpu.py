"""Every layout of a row over a warp, forward and backward, against the oracle.

A row of n 16-byte vectors takes the smallest power of two of lanes that holds it
(lanes past the row idle), and 2 or 4 vectors per lane above 32. The sizes are
the edges of each layout; one handle holds them all (one launch for tables of
several layouts), one holds a single size. Bag lengths mix one-lookup bags (whole
load groups of them take a path of their own), empty bags, bags that end inside
a group, and bags split across chunks; the tolerances are those of the other
forward and backward tests (1e-5 for fp32 sums, 2e-3 for half-precision rows).
"""

import pytest
import torch

from tests.helpers import (RTOL, assert_backward_matches, assert_forward_close, backward_reference,
                           forward_reference, inject_out_of_range, table_meta, without_lookups)

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
VECTORS = [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 31, 32, 33, 40, 64, 65, 128]


def _problem(vectors, dtype, seed, batch=150):
    g = torch.Generator().manual_seed(seed)
    per = 4 if dtype == torch.float32 else 8
    dims = [min(v * per, 512) for v in vectors]
    rows = [int(torch.randint(3, 400, (1,), generator=g)) for _ in dims]
    tables = [torch.randn(r, d, generator=g).to(dtype) for r, d in zip(rows, dims)]
    lens = []
    for _ in dims:
        x = torch.ones(batch, dtype=torch.int64)
        x[40:90] = torch.randint(0, 6, (50,), generator=g)
        x[90:-10] = torch.randint(0, 60, (max(batch - 100, 0),), generator=g)
        x[95 if batch > 110 else 5] = 700
        x[-10:] = 0  # trailing empty bags
        lens.append(x)
    lens = torch.cat(lens)
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64)
    off[1:] = torch.cumsum(lens, 0)
    ind = torch.cat([torch.randint(0, r, (int(off[(t + 1) * batch] - off[t * batch]),), generator=g)
                     for t, r in enumerate(rows)])
    w = torch.rand(ind.numel(), generator=g)
    go = torch.randn(batch, sum(dims), generator=g)
    return tables, ind, off, w, go, batch


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16])
@pytest.mark.parametrize("weighted,pooling", [(False, "sum"), (True, "mean")])
@pytest.mark.parametrize("vectors", [VECTORS, [3], [12], [31], [33], [128]], ids=str)
def test_forward_and_backward(vectors, dtype, weighted, pooling):
    from paper_2609_30656_gb300.tbe import TBE
    tables, ind, off, w, go, batch = _problem(vectors, dtype, 7 + len(vectors) + vectors[0])
    w = w if weighted else None
    mean = pooling == "mean"
    m = TBE([t.to(DEV) for t in tables], pooling=pooling, validate=True)
    dw = None if w is None else w.to(DEV)
    y = m.forward(ind.to(DEV), off.to(DEV), dw)
    g = m.backward(ind.to(DEV), off.to(DEV), go.to(DEV), dw)
    torch.cuda.synchronize()
    ref, scale = forward_reference(tables, batch, ind, off, w, mean)
    assert_forward_close(y, ref, scale, RTOL[dtype], what=f"{vectors} {dtype}")
    rows, dims = table_meta(tables)
    res, sc = backward_reference(rows, dims, batch, ind, off, go, w, mean)
    assert_backward_matches(g, res, sc, what=f"{vectors} {dtype}")


@pytest.mark.parametrize("vectors", [VECTORS, [12]], ids=str)
def test_out_of_range_lookups_among_single_lookup_bags(vectors):
    from paper_2609_30656_gb300.tbe import TBE
    tables, ind, off, _, go, batch = _problem(vectors, torch.float32, 31)
    bad_ind, bad = inject_out_of_range(tables, ind, off, batch, 32, frac=0.2)
    m = TBE([t.to(DEV) for t in tables], pooling="sum")
    y = m.forward(bad_ind.to(DEV), off.to(DEV))
    assert m.get_error() == 2  # reported, and the lookups add nothing
    g = m.backward(bad_ind.to(DEV), off.to(DEV), go.to(DEV))
    assert m.get_error() == 2
    kept_ind, kept_off, _ = without_lookups(bad_ind, off, None, bad, False)
    ref, scale = forward_reference(tables, batch, kept_ind, kept_off, None, False)
    assert_forward_close(y, ref, scale, RTOL[torch.float32], what="forward")
    rows, dims = table_meta(tables)
    res, sc = backward_reference(rows, dims, batch, kept_ind, kept_off, go, None, False)
    assert_backward_matches(g, res, sc, what="backward")


@pytest.mark.parametrize("batch", [100, 1200])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
def test_few_and_many_chunks_integer_tables(batch, weighted, dtype):
    # A forward with few chunks places them in the gather itself, one with many has a
    # kernel for it; integer values make every sum exact.
    import numpy as np
    from paper_2609_30656_gb300.tbe import TBE
    tables, ind, off, w, _, _ = _problem(VECTORS, dtype, 77, batch=batch)
    g = torch.Generator().manual_seed(78)
    tables = [torch.randint(-8, 9, t.shape, generator=g).to(dtype) for t in tables]
    w = torch.randint(0, 3, (ind.numel(),), generator=g).float() if weighted else None
    m = TBE([t.to(DEV) for t in tables], validate=True)
    y = m.forward(ind.to(DEV), off.to(DEV), None if w is None else w.to(DEV))
    ref, _ = forward_reference(tables, batch, ind, off, w, False)
    np.testing.assert_array_equal(y.cpu().double().numpy(), ref)
