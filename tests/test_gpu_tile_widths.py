"""Residue products at every tile width of the GEMM (32 to 256 columns): what
is put together is an integer, so a column's result has the same bits whatever
width its product ran at, alone and in a batch."""

import numpy as np
import pytest
import torch

from paper_1805_10121_gb300 import chase
from tests.test_gpu_rns import gauss, hermitian

pytestmark = pytest.mark.gpu

DEGREE = 4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


def filtered(h, v, split):
    fn = chase.chase_filter if v.is_complex() else chase.chase_filter_real
    return fn(h, v.clone(), [DEGREE] * v.shape[1], 1.6, -1.5, -0.9,
              precision=chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64)


# a block of 32 k columns takes tiles of 32 k; 300 rows: a second row tile, part filled
@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("real", [False, True])
def test_filter(split, real):
    h, v = hermitian(300, 3, real), gauss(300, 256, 4, real)
    want = filtered(h, v, split)
    for b in range(32, 256, 32):
        assert torch.equal(filtered(h, v[:, :b], split), want[:, :b])


@pytest.mark.parametrize("split", [False, True])
def test_batch(split):
    h, v = hermitian(300, 5, False), gauss(300, 256, 6, False)
    want = filtered(h, v, split)
    for b in range(32, 257, 32):
        x = [v[:, :b].clone()]
        chase.chase_filter_batched([h], x, [np.full(b, DEGREE, dtype=np.int32)], [1.6], [-1.5], [-0.9],
                                   precision=chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64)
        assert torch.equal(x[0], want[:, :b])
