"""Lanczos on the residue planes of H (from N^2 r = 4e6 on) and on the
few-column kernel, through solves on both sides of that line."""

import numpy as np
import pytest
import torch

import oracle
from paper_1805_10121_gb300 import chase, synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


def solve(n, nev, nex, seed, runs, **opts):
    lam = synth.spectrum_uniform(n, seed, device=DEV)
    h = synth.hermitian_dft(lam, seed + 1)
    v = synth.gaussian_block(n, nev + nex, seed + 2, device=DEV)
    s = synth.gaussian_block(n, 1 + runs, seed + 3, device=DEV)
    o = chase.chase_opts_default(num_lanczos=runs, **opts)
    st, ritz, res, stats = chase.chase_solve(h, nev, nex, 1e-10, v, s, opts=o)
    assert st == chase.CHASE_OK
    lam = lam.cpu().numpy()
    top = np.abs(lam).max()
    assert np.max(np.abs(ritz[:nev] - lam[:nev])) <= 1e-10 * top
    r = oracle.residuals(h.cpu().numpy(), v.cpu().numpy()[:, :nev], ritz[:nev])
    assert np.all(r <= 1.05e-10 * top)
    # the bounds: above the largest eigenvalue, by no more than the spectrum
    assert lam[-1] <= stats["b_sup"] <= lam[-1] + (lam[-1] - lam[0])


@pytest.mark.parametrize("n,runs", [(880, 4), (900, 4), (1300, 1), (1500, 1)])
@pytest.mark.parametrize("precision", [chase.CHASE_FP64, chase.CHASE_SPLIT_BF16, chase.CHASE_SPLIT_BF16_RR])
def test_either_side(n, runs, precision):
    solve(n, 40, 16, n, runs, precision=precision)
