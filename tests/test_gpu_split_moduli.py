"""Where split products take 12 moduli (operands rounded to 2^-52 of a norm)
instead of 11 (2^-48): H Q of CHASE_SPLIT_BF16_RR, and filters of a few steps on
long sums (K = 2 N complex, N real, above 16384), where one product's rounding
would exceed that of the digit splits these stand for.

The counters tell the moduli: a product executes 2 N^2 FLOPs a plane and column,
two planes a modulus when complex, beside 8 N^2 (2 N^2 real) algorithmic ones."""

import pytest
import torch

from paper_1805_10121_gb300 import chase, synth
from tests.test_gpu_memory import timed
from tests.test_gpu_rns import U, reference

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


def hermitian(n, real):
    g = torch.Generator(device="cuda").manual_seed(n)
    a = torch.randn(n, n, dtype=torch.float64 if real else torch.complex128, device="cuda", generator=g)
    a += a.conj().t().clone()
    return a.mul_(1.0 / (4.0 * n ** 0.5)).t()


@pytest.mark.parametrize("n,real,degrees,moduli", [
    (8192, False, [2] * 8, 11), (8193, False, [2] * 8, 12), (8193, False, [8] * 7 + [6], 12),
    (8193, False, [8] * 8, 11), (8193, True, [2] * 8, 11), (16385, True, [4] * 8, 12)])
def test_filter(n, real, degrees, moduli):
    h = hermitian(n, real)
    v = torch.randn(8, n, dtype=h.dtype, device="cuda", generator=torch.Generator("cuda").manual_seed(1)).t()
    got = v.clone()
    fn = chase.chase_filter_real if real else chase.chase_filter
    _, share = timed(chase.CHASE_TIMED_SPLIT_PRODUCT,
                     lambda: fn(h, got, degrees, 1.6, -1.5, -0.9, precision=chase.CHASE_SPLIT_BF16))
    assert share == pytest.approx(moduli if real else moduli / 2.0)
    m = degrees[-1]
    ref = reference(h, v[:, -1:], m, 1.6, -1.5, -0.9)
    e = float(torch.linalg.norm(got[:, -1:] - ref) / torch.linalg.norm(ref))
    # operands to 2^-L of a norm (test_gpu_rns.py)
    assert e <= 8 * m * ((2 * n) ** 0.5 * 2.0 ** -(48 if moduli == 11 else 52) + 8 * U + (2 * n) ** 0.5 * U)


@pytest.mark.parametrize("batched", [False, True])
def test_rayleigh_ritz_product(batched):
    n, nev, nex = 400, 20, 8
    lam = synth.spectrum_uniform(n, 3, device="cuda")
    h, v = synth.hermitian_dft(lam, 4), synth.gaussian_block(n, nev + nex, 5, device="cuda")
    s = synth.gaussian_block(n, 5, 6, device="cuda")
    o = chase.chase_opts_default(precision=chase.CHASE_SPLIT_BF16_RR)

    def solve():
        if batched:
            chase.chase_solve_batched([h], [nev], [nex], 1e-10, [v], [s], opts=o)
        else:
            chase.chase_solve(h, nev, nex, 1e-10, v, s, opts=o)
    _, share = timed(chase.CHASE_TIMED_SPLIT_PRODUCT, solve)
    assert share == pytest.approx(6.0)
