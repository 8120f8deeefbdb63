"""The FM cross term at the edges of its block shapes: one sample or many per block,
every number of fields held per thread (2, 4, 8, 16) and the loop above that, thread
rows that are not a power of two, and a row stride wider than the row; and batch
replication at the edges of its blocks."""

import numpy as np
import pytest
import torch

import oracle
from tests.test_fm_gpu import _check_fm

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("T,D,B", [(1, 4, 1), (2, 4, 1000), (300, 4, 3), (5, 20, 129), (26, 48, 64), (27, 96, 9),
                                   (100, 128, 7), (100, 256, 5), (16, 512, 4), (17, 512, 4), (32, 512, 4), (33, 512, 4),
                                   (64, 64, 33), (257, 64, 2), (3, 508, 6)])
def test_shapes(T, D, B):
    g = torch.Generator(device=DEV).manual_seed(T * D + B)
    y = torch.randn(B, T * D + 8, generator=g, device=DEV)
    _check_fm(y[:, :T * D].contiguous(), T, torch.randn(B, generator=g, device=DEV))
    from paper_2609_30656_gb300 import tbe
    wide = tbe.fm_forward(y[:, :T * D], T)  # the same samples, further apart
    assert torch.equal(wide, tbe.fm_forward(y[:, :T * D].contiguous(), T))


@pytest.mark.parametrize("T,B,factor", [(1, 1, 1), (3, 85, 2), (2, 256, 5), (700, 3, 3), (2049, 2, 2), (4, 64, 300)])
@pytest.mark.parametrize("dtype", [torch.int32, torch.int64])
def test_replicate(T, B, factor, dtype):
    from paper_2609_30656_gb300 import tbe
    g = torch.Generator().manual_seed(T + B)
    lens = torch.randint(0, 9, (T * B,), generator=g)
    lens[: B] = 0
    off = torch.zeros(T * B + 1, dtype=dtype)
    off[1:] = torch.cumsum(lens, 0)
    ind = torch.randint(0, 1000, (int(off[-1]),), generator=g).to(dtype)
    w = torch.rand(ind.numel(), generator=g)
    got = tbe.replicate_batch(ind.to(DEV), off.to(DEV), w.to(DEV), T, factor)
    for a, b in zip(got, oracle.replicate_kjt(ind, off, w, T, factor)):
        np.testing.assert_array_equal(a.cpu().numpy(), b)


def test_replicate_as_often_as_32_bits_count():
    from paper_2609_30656_gb300 import tbe
    F = 2 ** 31 - 1  # one bag of one lookup: the most copies that the entry point takes
    ind, off = torch.tensor([5], dtype=torch.int32, device=DEV), torch.tensor([0, 1], dtype=torch.int32, device=DEV)
    got_ind, got_off, _ = tbe.replicate_batch(ind, off, None, 1, F)
    assert int(got_off[0]) == 0 and int(got_off[-1]) == F
    step = 1 << 28
    for a in range(0, F, step):
        b = min(a + step, F)
        assert torch.equal(got_off[a:b], torch.arange(a, b, dtype=torch.int32, device=DEV))
        assert bool((got_ind[a:b] == 5).all())
