"""Products in residue arithmetic on the tensor cores (csrc/rns.cu) through
the filter and residual entry points, at the edges of their tiles (256 rows
and 32 ... 256 columns per CTA pair, 64-wide K stages, chunks of 256 to 448
K), against plain 64-bit torch products.

Tolerance.  The operands are rounded to 2^-L of the 2-norm of a row of H or a
column of X (L = 60 in FP64 mode, 48 in split mode), so one product is off by
at most sqrt(2 K) 2^-L (|H| + |X| rounding, relative to norm products), and
by the FP64 roundings of the epilogue, a few 2^-53.  A degree-m filter adds m
of them; its values stay within a factor of about 2 m of its input's norm
(Chebyshev recurrence).  The bars below allow 8 m that sum, and 8 m u more
for the recurrence's FP64 operations on both sides."""

import numpy as np
import pytest
import torch

from paper_1805_10121_gb300 import chase

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


def gauss(n, b, seed, real):
    g = torch.Generator(device="cpu").manual_seed(seed)
    x = torch.randn(b, n, dtype=torch.float64, generator=g)
    if not real:
        x = torch.complex(x, torch.randn(b, n, dtype=torch.float64, generator=g))
    return x.to(DEV).t()


def hermitian(n, seed, real):
    a = gauss(n, n, seed, real)
    h = (a + a.conj().t()) / (4.0 * (n ** 0.5))  # spectrum inside [-1.5, 1.5]
    return h.t().contiguous().t()


def reference(h, v, m, b_sup, mu1, mu_nn):
    c, e = 0.5 * (b_sup + mu_nn), 0.5 * (b_sup - mu_nn)
    s1 = sigma = e / (mu1 - c)
    prev, cur = v, (s1 / e) * (h @ v - c * v)
    for _ in range(2, m + 1):
        tau = 1.0 / (2.0 / s1 - sigma)
        prev, cur = cur, (2.0 * tau / e) * (h @ cur - c * cur) - tau * sigma * prev
        sigma = tau
    return cur


def bar(n, m, split):
    return 8 * m * ((2 * n) ** 0.5 * 2.0 ** -(48 if split else 60) + 8 * U + (2 * n) ** 0.5 * U)


def err(x, y):
    return float((torch.linalg.norm(x - y, dim=0) / torch.linalg.norm(y, dim=0)).max())


@pytest.mark.parametrize("n,b", [(128, 7), (129, 32), (255, 33), (256, 64), (257, 97), (320, 160),
                                 (449, 225), (512, 257), (1025, 40), (2050, 513)])
@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("real", [False, True])
def test_filter_at_tile_edges(n, b, split, real):
    h, v, m = hermitian(n, n + b, real), gauss(n, b, n - b, real), 6
    ref = reference(h, v, m, 1.6, -1.5, -0.9)
    got = v.clone()
    fn = chase.chase_filter_real if real else chase.chase_filter
    fn(h, got, [m] * b, 1.6, -1.5, -0.9,
       precision=chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64)
    assert err(got, ref) <= bar(n, m, split)


@pytest.mark.parametrize("n", [700, 1900])
def test_sums_without_cancellation(n):
    # every entry of every product has one sign: the accumulators reach the
    # most that a chunk allows
    h = torch.ones(n, n, dtype=torch.complex128, device=DEV).t() / n
    v = torch.ones(9, n, dtype=torch.complex128, device=DEV).t().clone(memory_format=torch.preserve_format)
    ref = reference(h, v, 4, 1.6, -1.5, -0.9)
    chase.chase_filter(h, v, [4] * 9, 1.6, -1.5, -0.9)
    assert err(v, ref) <= bar(n, 4, False)


@pytest.mark.parametrize("scale", [1e-290, 1e-160, 1e120])
def test_residuals_of_extreme_columns(scale):
    # columns whose squares under- or overflow, and a zero column
    n, b = 300, 12
    h, v = hermitian(n, 3, False), gauss(n, b, 4, False).clone()
    f = torch.full((b,), scale, dtype=torch.float64, device=DEV)
    f[::2] = 1.0
    v = (v * f[None, :]).t().contiguous().t()
    v[:, 5] = 0.0
    r = torch.from_numpy(chase.chase_residuals(h, v, np.zeros(b))).to(DEV)
    w = h @ v
    for j in range(b):
        a = torch.linalg.norm(w[:, j] / f[j]) * f[j] if scale > 1e-200 or j % 2 == 0 else None
        if j == 5:
            assert float(r[j]) == 0.0
        elif a is not None and (scale > 1e-150 or j % 2 == 0):  # the norm's own squares fit
            assert abs(float(r[j]) - float(a)) <= 1e-12 * float(a)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_entries_reach_the_result(bad):
    # residuals take any input: a bad column poisons its own residual, a bad
    # row of H every residual
    n, b = 300, 12
    h, v = hermitian(n, 5, False), gauss(n, b, 6, False).clone()
    w = v.clone()
    w[17, 3] = bad
    r = chase.chase_residuals(h, w, np.zeros(b))
    good = chase.chase_residuals(h, v, np.zeros(b))
    assert not np.isfinite(r[3])
    assert np.array_equal(np.delete(r, 3), np.delete(good, 3))
    h = h.clone()
    h[7, 9] = bad
    h[9, 7] = bad
    assert not np.any(np.isfinite(chase.chase_residuals(h, v, np.zeros(b))))
