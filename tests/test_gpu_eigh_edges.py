"""The projected eigensolve at the sizes where its code changes (csrc/
eigh_refine.cu: 8 refined at all, 32 / 64 / 96 rows per lane of the one-block
Jacobi solve, 97 the library's FP32 solver), complex through Rayleigh-Ritz
with clustered and multiple eigenvalues, and real through a solve.

Tolerance: as in test_gpu_eigh.py."""

import numpy as np
import pytest
import torch

from paper_1805_10121_gb300 import chase
from tests.test_gpu_eigh import DEV, check, spectrum, unitary

pytestmark = pytest.mark.gpu

EDGES = [8, 9, 31, 32, 63, 64, 65, 95, 96, 97]
KINDS = ["plain", "double", "constant", "gap1e-7", "gap1e-13", "many close"]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


@pytest.mark.parametrize("p", EDGES)
@pytest.mark.parametrize("kind", KINDS)
def test_complex(p, kind):
    n = 240
    rng = np.random.default_rng(p)
    lam = spectrum(kind, p, rng)
    w = unitary(n, p, rng)
    h = (w * lam) @ w.conj().T
    check(0.5 * (h + h.conj().T), w @ unitary(p, p, rng), np.sort(lam))


@pytest.mark.parametrize("p", EDGES)
def test_real(p):
    # there is no real Rayleigh-Ritz entry: through a solve, whose first
    # iteration projects all p = nev + nex columns
    n, nex = 400, max(2, p // 4)
    rng = np.random.default_rng(100 + p)
    lam = np.sort(rng.uniform(-1.0, 1.0, n))
    q = np.linalg.qr(rng.standard_normal((n, n)))[0]
    h = (q * lam) @ q.T
    hd = torch.from_numpy(0.5 * (h + h.T)).to(DEV).t().contiguous().t()
    v = torch.from_numpy(rng.standard_normal((p, n))).to(DEV).t()
    s = torch.from_numpy(rng.standard_normal((5, n))).to(DEV).t()
    st, ritz, _, _ = chase.chase_solve_real(hd, p - nex, nex, 1e-10, v, s)
    assert st == chase.CHASE_OK
    assert np.max(np.abs(ritz[:p - nex] - lam[:p - nex])) <= 1e-10
    x = v.cpu().numpy()[:, :p - nex]
    assert np.linalg.norm(x.T @ x - np.eye(p - nex)) <= 20 * (p + n ** 0.5) * 2.0 ** -53
    assert np.max(np.linalg.norm(h @ x - x * ritz[:p - nex], axis=0)) <= 1.05e-10
