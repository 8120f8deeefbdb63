"""The FM cross term at the edges of its block shapes: one sample or many per block,
every number of fields held per thread (2, 4, 8, 16) and the loop above that, thread
rows that are not a power of two, and a row stride wider than the row; at the edges of a
warp's: the fewest vectors that it takes, every number of steps that it holds (2, 4, 8, 16
for each 32 vectors of a field) and the loop above that; and batch replication at the edges
of its blocks."""

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


# a warp per sample: 15 to 21 vectors, and steps at and above 2, 4, 8, 16 and 48 for fields
# of 1 to 128 vectors; below and at the batch from which the forward loops,
# and at the size from which it does not
WARP = [(15, 4, 9), (16, 4, 9), (17, 4, 9), (10, 8, 70), (20, 4, 9), (21, 4, 9), (7, 12, 8), (3, 28, 9), (64, 4, 9), (65, 4, 9), (129, 4, 3), (257, 4, 3),
        (513, 4, 2), (48, 36, 1024), (48, 36, 1023), (32, 64, 7), (33, 64, 1024), (96, 64, 1024), (97, 64, 1024),
        (2, 128, 5), (3, 128, 5), (5, 100, 5), (9, 128, 5), (16, 128, 5), (17, 128, 1024), (48, 128, 1100), (49, 128, 1024),
        (2, 132, 3), (2, 256, 3), (3, 256, 3), (5, 256, 3), (8, 256, 3), (9, 256, 1024), (24, 192, 1024), (25, 192, 1024),
        (1, 260, 3), (2, 384, 3), (3, 384, 3), (5, 384, 3), (6, 384, 1024), (16, 300, 1024), (17, 384, 1024),
        (1, 512, 3), (2, 512, 3), (3, 512, 3), (4, 388, 3), (5, 512, 1024), (12, 512, 1024), (13, 512, 1024), (24, 128, 10922),
        (24, 128, 10923)]


@pytest.mark.parametrize("T,D,B", WARP)
def test_warp_shapes(T, D, B):
    test_shapes(T, D, B)


def test_forward_takes_as_long_whatever_the_fields():
    """64 MB of small samples against 64 MB of large ones (1.2 times as long; 3.3 times when a
    block took each few small samples)."""
    from paper_2609_30656_gb300 import tbe
    from tests.test_split_segments_gpu import _times
    took = []
    for T, D in ((100, 8), (26, 128)):
        y = torch.randn((64 << 20) // (4 * T * D), T * D, device=DEV)
        out = torch.empty(y.shape[0], device=DEV)

        def call():
            for _ in range(8):
                tbe.fm_forward(y, T, out=out)
        took.append(_times(call))
    assert took[0] < 2 * took[1], took


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
