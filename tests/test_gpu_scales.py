"""Residue planes of H with one scale for all rows (one plane per modulus, the
second operand a transposed tile of it) and with a scale per row (two planes):
both sides of the rule that chooses, at the edges of the 64 x 64 tiles that
slice H and of the product's 256-row tiles, alone and mixed in a batch.

Tolerance: as in test_gpu_rns.py, operands rounded to 2^-L of a norm (L = 60
or 48; a common scale costs a row at most one bit) and FP64 roundings, for
each of the m products of a filter whose values stay within 2 m of the
input's norm; 16 m allows that bit."""

import numpy as np
import pytest
import torch

from paper_1805_10121_gb300 import chase
from tests.test_gpu_rns import DEV, U, gauss, hermitian, reference

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


def bar(n, m, split):
    return 16 * m * ((2 * n) ** 0.5 * 2.0 ** -(48 if split else 60) + 8 * U + (2 * n) ** 0.5 * U)


def matrix(n, seed, kind):
    h = hermitian(n, seed, False).clone()
    if kind == "graded":  # rows over three decades: a scale per row
        d = torch.logspace(0.0, -1.5, n, dtype=torch.float64, device=DEV)
        h = d[:, None] * h * d[None, :]
    elif kind == "diagonal":  # no row has anything beside its diagonal
        h = torch.diag(torch.diagonal(h).real).to(torch.complex128)
    elif kind == "zero rows":
        h[n // 3, :] = 0.0
        h[:, n // 3] = 0.0
    elif kind == "rounded":  # Hermitian up to rounding
        h = h * (1.0 + U * torch.randn(n, n, dtype=torch.float64, device=DEV))
    return h.t().contiguous().t()


def err(x, y):
    return float((torch.linalg.norm(x - y, dim=0) / torch.linalg.norm(y, dim=0)).max())


KINDS = ["plain", "graded", "diagonal", "zero rows", "rounded"]


# with one scale the planes are halved above 64 MB of them: N = 1069 (FP64) and
# 1206 (split); the sizes below 1000 take two planes in any case
@pytest.mark.parametrize("n,b", [(129, 33), (449, 97), (1025, 20), (1089, 9), (1216, 65), (1279, 40), (1281, 225),
                                 (1409, 8), (2050, 150)])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("split", [False, True])
def test_filter(n, b, kind, split):
    h, v, m = matrix(n, n + b, kind), gauss(n, b, n - b, False), 6
    ref = reference(h, v, m, 1.6, -1.5, -0.9)
    got = v.clone()
    chase.chase_filter(h, got, [m] * b, 1.6, -1.5, -0.9,
                       precision=chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64)
    assert err(got, ref) <= bar(n, m, split)


@pytest.mark.parametrize("n,b", [(700, 70), (1537, 10), (1600, 130)])
@pytest.mark.parametrize("kind", KINDS)
def test_filter_single_precision(n, b, kind):
    h, v, m = matrix(n, n + b, kind), gauss(n, b, n - b, False), 6
    h, v = (x.to(torch.complex64).t().contiguous().t() for x in (h, v))
    ref = reference(h.to(torch.complex128), v.to(torch.complex128), m, 1.6, -1.5, -0.9)
    chase.chase_filter_c32(h, v, [m] * b, 1.6, -1.5, -0.9)
    # operands to 2^-30, results stored in FP32 after each of the m steps
    assert err(v, ref) <= 16 * m * ((2 * n) ** 0.5 * 2.0 ** -30 + 8 * 2.0 ** -24)


@pytest.mark.parametrize("split", [False, True])
def test_batch_of_both_kinds(split):
    shapes = [(1000, 20), (129, 9), (513, 64), (64, 5), (700, 40), (1, 1), (1025, 31)]
    hs = [matrix(n, 7 * i, KINDS[i % len(KINDS)]) for i, (n, b) in enumerate(shapes)]
    vs = [gauss(n, b, 100 + i, False).clone() for i, (n, b) in enumerate(shapes)]
    degs = [np.full(b, 4 + 2 * (i % 2), dtype=np.int32) for i, (n, b) in enumerate(shapes)]
    refs = [reference(h, v, int(d[0]), 1.6, -1.5, -0.9) for h, v, d in zip(hs, vs, degs)]
    chase.chase_filter_batched(hs, vs, degs, [1.6] * 7, [-1.5] * 7, [-0.9] * 7,
                               precision=chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64)
    for (n, b), v, ref, d in zip(shapes, vs, refs, degs):
        assert err(v, ref) <= bar(max(n, 64), int(d[0]), split)


# real H holds one triangle from N = 1537 (FP64), 1728 (split) and 2150 (FP32) on
@pytest.mark.parametrize("n,b", [(1100, 30), (1537, 33), (1791, 65), (1793, 9), (2047, 17), (2305, 130)])
@pytest.mark.parametrize("kind", ["plain", "graded", "rounded"])
@pytest.mark.parametrize("field,split", [("f64", False), ("f64", True), ("f32", False)])
def test_real_filter(n, b, kind, field, split):
    g = hermitian(n, n + b, True).clone()
    if kind == "graded":
        d = torch.logspace(0.0, -1.5, n, dtype=torch.float64, device=DEV)
        g = d[:, None] * g * d[None, :]
    elif kind == "rounded":
        g = g * (1.0 + U * torch.randn(n, n, dtype=torch.float64, device=DEV))
    dt = torch.float64 if field == "f64" else torch.float32
    h, v = (x.to(dt).t().contiguous().t() for x in (g, gauss(n, b, n - b, True)))
    ref = reference(h.double(), v.double(), 6, 1.6, -1.5, -0.9)
    if field == "f64":
        chase.chase_filter_real(h, v, [6] * b, 1.6, -1.5, -0.9,
                                precision=chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64)
        assert err(v, ref) <= bar(n, 6, split)
    else:
        chase.chase_filter_f32(h, v, [6] * b, 1.6, -1.5, -0.9)
        assert err(v.double(), ref) <= 16 * 6 * ((2 * n) ** 0.5 * 2.0 ** -30 + 8 * 2.0 ** -24)
