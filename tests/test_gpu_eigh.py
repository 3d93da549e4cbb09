"""The projected eigensolve of Rayleigh-Ritz (csrc/eigh_refine.cu: an FP32
solve refined by products) on both sides of the size where it takes over, with
spectra that a refinement can get wrong: clusters far below FP32 resolution,
exact multiplicities, one value only, and extreme scales.

Tolerance.  An FP64 eigensolver's backward error, a few p u ||G||, with the
roundings of the N-long products that form G and the residuals."""

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


def unitary(n, p, rng):
    return np.linalg.qr(rng.standard_normal((n, p)) + 1j * rng.standard_normal((n, p)))[0]


def spectrum(kind, p, rng):
    lam = np.sort(rng.standard_normal(p))
    if kind == "shifted":
        lam = 1000.0 + lam
    elif kind == "double":
        lam[1::2] = lam[0:2 * (p // 2):2]
    elif kind == "constant":
        lam[:] = -0.7
    elif kind.startswith("gap"):
        m = p // 3
        k = min(6, p - m)
        lam[m:m + k] = lam[m] + float(kind[3:]) * np.arange(k)
    elif kind == "many close":
        lam = 1e-8 * np.arange(p) + (np.arange(p) >= p // 2)
    return lam


@pytest.mark.parametrize("p", [7, 23, 24, 33, 70, 129, 197])
@pytest.mark.parametrize("kind", ["plain", "shifted", "double", "constant", "gap1e-5", "gap1e-7", "gap1e-9",
                                  "gap1e-13", "many close"])
def test_spectra(p, kind):
    n = 320
    rng = np.random.default_rng(p)
    lam = spectrum(kind, p, rng)
    w = unitary(n, p, rng)
    h = (w * lam) @ w.conj().T
    h = 0.5 * (h + h.conj().T)
    q = w @ unitary(p, p, rng)
    check(h, q, np.sort(lam))


@pytest.mark.parametrize("scale", [1e-100, 1e-20, 1e20, 1e100])
def test_scales(scale):
    n, p = 300, 60
    rng = np.random.default_rng(3)
    lam = np.sort(rng.standard_normal(p)) * scale
    w = unitary(n, p, rng)
    h = (w * lam) @ w.conj().T
    check(0.5 * (h + h.conj().T), w @ unitary(p, p, rng), lam)


def check(h, q, lam):
    n, p = q.shape
    qd = torch.from_numpy(q).to(DEV).t().contiguous().t()
    ritz, resid = chase.chase_rayleigh_ritz(torch.from_numpy(h).to(DEV).t().contiguous().t(), qd)
    x = qd.cpu().numpy()
    top = np.max(np.abs(lam))
    bar = 20 * (p + n ** 0.5) * U * top
    assert np.all(np.diff(ritz) >= 0)
    assert np.max(np.abs(ritz - lam)) <= bar
    assert np.linalg.norm(x.conj().T @ x - np.eye(p)) <= 20 * (p + n ** 0.5) * U
    assert np.max(np.linalg.norm(h @ x - x * ritz, axis=0)) <= bar
    assert np.max(resid) <= bar
