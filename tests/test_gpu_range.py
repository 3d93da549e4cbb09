"""Filters whose diagonal term alpha (H_rr - shift) is far outside FP32's range
(bounds that do not bracket the spectrum): the products whose constants carry
parts in FP32 must still give what 64-bit arithmetic gives.

Tolerance: every row of the result is dominated by the huge entry's row or
column, to which the operands' rounding (2^-60 of a norm; single precision
2^-30, results stored in FP32) is relative."""

import numpy as np
import pytest
import torch

from paper_1805_10121_gb300 import chase
from tests.test_gpu_chain import FILTER, TYPE
from tests.test_gpu_rns import gauss, hermitian, reference

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


@pytest.mark.parametrize("n,field,huge,tiny,bounds,tol", [
    (130, "c128", 190, 0, (1.6, -1.5, -0.9), 1e-11),
    (130, "f64", 190, 0, (1.6, -1.5, -0.9), 1e-11),
    (2100, "c128", 190, 0, (1.6, -1.5, -0.9), 1e-11),  # not chained
    (130, "c64", 127, -139, (1.6, 1.4, 1.5), 1e-2),    # inputs denormal: 10 bits
    (130, "f32", 127, -139, (1.6, 1.4, 1.5), 1e-2),
])
def test_one_huge_diagonal_entry(n, field, huge, tiny, bounds, tol):
    real = field in ("f64", "f32")
    h = hermitian(n, 3, real).clone()
    h[5, 5] = 1.1 * 2.0 ** huge
    h = h.to(TYPE[field]).t().contiguous().t()
    v = gauss(n, 8, 4, real) * 2.0 ** tiny
    if not tiny:
        v[5] *= 2.0 ** -120  # the product, 2^70, is still the largest of its column
    v = v.to(TYPE[field]).t().contiguous().t()
    up = torch.float64 if real else torch.complex128
    ref = reference(h.to(up), v.to(up), 2, *bounds)
    if field in ("c64", "f32"):
        assert float(ref.abs().max()) < 3e38
    FILTER[field](h, v, [2] * 8, *bounds)
    got = v.to(up)
    assert torch.isfinite(torch.view_as_real(got) if not real else got).all()
    e = torch.linalg.norm(got - ref, dim=1) / torch.linalg.norm(ref, dim=1)
    assert float(e[5]) <= tol
    assert float(e.max()) <= 100 * tol
