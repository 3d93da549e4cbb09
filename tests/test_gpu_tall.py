"""Cholesky QR and Rayleigh-Ritz on tall blocks in residue arithmetic, at the
edges of their kernels: 16-wide Cholesky blocks, 32-row and 64-wide slicing
tiles, 256-row and 32 ... 256-column product tiles, and the smallest sizes
that take the residue path (N = 128, 7 columns) and the largest that do not.

Tolerance.  Products round their operands to 2^-60 of a vector's norm, below
FP64 rounding, so the bars are those of FP64 Cholesky QR applied twice:
orthonormality to a few b u, and the factor R = Q^H V unique for a positive
diagonal, hence Q within about cond(V) b u of Householder's."""

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


def gauss(n, b, seed):
    g = torch.Generator(device="cpu").manual_seed(seed)
    return torch.complex(torch.randn(b, n, dtype=torch.float64, generator=g),
                         torch.randn(b, n, dtype=torch.float64, generator=g)).t()


def on_device(x):
    return x.to(DEV).t().contiguous().t()


def householder(v):
    q, r = np.linalg.qr(v)
    d = np.diag(r)
    return q * (d / np.abs(d))[None, :], float(np.linalg.cond(r))


@pytest.mark.parametrize("n,b,nconv", [(127, 9, 5), (128, 6, 4), (128, 7, 0), (129, 16, 1), (200, 17, 3),
                                       (257, 32, 33), (300, 33, 16), (449, 48, 7), (513, 100, 64),
                                       (1025, 65, 257), (1500, 255, 0), (2050, 300, 31)])
@pytest.mark.parametrize("scales", [0.0, 6.0])
def test_orthonormalize(n, b, nconv, scales):
    v = gauss(n, b, n + b).numpy() * np.logspace(0.0, -scales, b)[None, :]
    y = np.linalg.qr(gauss(n, nconv, n).numpy())[0] if nconv else np.zeros((n, 0), complex)
    v = v + 0.3 * y @ (y.conj().T @ v)
    ref = v.copy()
    for _ in range(2):
        ref = ref - y @ (y.conj().T @ ref)
    ref, cond = householder(ref / np.linalg.norm(ref, axis=0))
    yd, vd = on_device(torch.from_numpy(y)), on_device(torch.from_numpy(v))
    q = chase.chase_orthonormalize(yd, vd).cpu().numpy()
    assert np.linalg.norm(q.conj().T @ q - np.eye(b)) <= 20 * (b + n ** 0.5) * U
    if nconv:
        assert np.linalg.norm(y.conj().T @ q) <= 20 * (b + nconv + n ** 0.5) * U
    assert np.linalg.norm(q - ref) <= 20 * cond * (b + nconv + n ** 0.5) * U


@pytest.mark.parametrize("n,b", [(128, 7), (300, 33), (700, 129)])
def test_rank_deficient_block_breaks_down(n, b):
    v = gauss(n, b, 1).numpy()
    v[:, b - 1] = 0.0
    y = np.zeros((n, 0), complex)
    with pytest.raises(Exception):
        chase.chase_orthonormalize(on_device(torch.from_numpy(y)), on_device(torch.from_numpy(v)))


@pytest.mark.parametrize("n,b", [(127, 9), (128, 7), (300, 33), (513, 100), (1100, 258)])
def test_rayleigh_ritz(n, b):
    a = gauss(n, n, 3 * n).numpy()
    h = (a + a.conj().T) / (4.0 * n ** 0.5)
    q, _ = householder(gauss(n, b, n - b).numpy())
    lam, w = np.linalg.eigh(q.conj().T @ h @ q)
    qd = on_device(torch.from_numpy(q))
    ritz, resid = chase.chase_rayleigh_ritz(on_device(torch.from_numpy(h)), qd)
    assert np.max(np.abs(ritz - lam)) <= 20 * (b + n ** 0.5) * U
    x = q @ w
    res = np.linalg.norm(h @ x - x * lam, axis=0)
    assert np.max(np.abs(resid - res)) <= 50 * (b + n ** 0.5) * U / max(np.min(np.diff(lam)), 1e-6)
    x = qd.cpu().numpy()
    assert np.linalg.norm(x.conj().T @ x - np.eye(b)) <= 20 * (b + n ** 0.5) * U


@pytest.mark.parametrize("n,b", [(300, 33), (700, 129)])
@pytest.mark.parametrize("decades", [0, 2, 4, 5])
def test_second_pass_near_and_far_from_the_identity(n, b, decades):
    # the first pass leaves cond(V)^2 u: below 1e-8 the second factor is its
    # first-order form, above it the whole elimination
    rng = np.random.default_rng(n + decades)
    w = np.linalg.qr(rng.standard_normal((b, b)) + 1j * rng.standard_normal((b, b)))[0]
    v = (householder(gauss(n, b, n).numpy())[0] * np.logspace(0.0, -decades, b)[None, :]) @ w
    ref, cond = householder(v)
    q = chase.chase_orthonormalize(None, on_device(torch.from_numpy(v))).cpu().numpy()
    assert np.linalg.norm(q.conj().T @ q - np.eye(b)) <= 20 * (b + n ** 0.5) * U
    assert np.linalg.norm(q - ref) <= 20 * cond * (b + n ** 0.5) * U
