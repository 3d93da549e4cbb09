"""Calls whose workspace does not hold all residue planes of H: fewer moduli
resident (H sliced anew for every product), fewer columns at a time, and, for
products at FP64 accuracy, the FP64 pipe.  The shortage is made on the host, by
chase_workspace_limit.

Tolerance: as in test_gpu_scales.py, whichever way the product was made (an
FP64 GEMM's n u is below its bar)."""

import contextlib

import numpy as np
import pytest
import torch

from paper_1805_10121_gb300 import chase, synth
from tests.test_gpu_chain import FILTER, TYPE, bar
from tests.test_gpu_rns import DEV, U, gauss, hermitian, reference
from tests.test_gpu_scales import err

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


@contextlib.contextmanager
def limit(nbytes):
    chase.chase_workspace_limit(nbytes)
    try:
        yield
    finally:
        chase.chase_workspace_limit(0)


def timed(kind, call):
    """The launches and the executed share of the FLOPs of call's products."""
    chase.chase_kernel_timing(True)
    try:
        call()
        k = chase.chase_kernel_timing_read(kind)
    finally:
        chase.chase_kernel_timing(False)
    return k["launches"], k["tensor_flops"] / k["flops"] if k["flops"] else 0.0


# N = 1200, 40 columns, complex, FP64: 41 MB of planes, 5 MB for the block, 11 MB in reserve
LIMITS = [1, 6, 17, 20, 28, 40, 0]


@pytest.mark.parametrize("field", ["c128", "f64", "c64", "f32"])
def test_filter(field):
    real, m = field in ("f64", "f32"), 6
    n, b = 1200, 40
    h, v = (x.to(TYPE[field]).t().contiguous().t() for x in (hermitian(n, 1, real), gauss(n, b, 2, real)))
    up = torch.float64 if real else torch.complex128
    ref = reference(h.to(up), v.to(up), m, 1.6, -1.5, -0.9)
    ways = set()
    for mb in LIMITS:
        got = v.clone()
        with limit(mb * MB):
            launches, share = timed(chase.CHASE_TIMED_FP64_PRODUCT,
                                    lambda: FILTER[field](h, got, [m] * b, 1.6, -1.5, -0.9))
        ways.add((launches, share))
        assert err(got.to(up), ref) <= bar(n, m, field, False)
    if field == "c128":  # 28 planes of 2 N^2 b beside 8 N^2 b, or the 3M form
        assert (m, 7.0) in ways and (m, 0.75) in ways
        assert any(s == 7.0 and k > m for k, s in ways)


@pytest.mark.parametrize("classes", [[7], [3], [3, 4, 7]])
def test_split_filter(classes):
    n, b, m = 1200, 40, 6
    h, v = hermitian(n, 3, False), gauss(n, b, 4, False)
    slices = [classes[i % len(classes)] for i in range(b)]
    ref = reference(h, v, m, 1.6, -1.5, -0.9)
    ways = set()
    for mb in (11, 14, 24, 48, 0):
        got = v.clone()
        with limit(mb * MB):
            ways.add(timed(chase.CHASE_TIMED_SPLIT_PRODUCT,
                           lambda: chase.chase_filter_mixed(h, got, [m] * b, slices, 1.6, -1.5, -0.9))[0])
        for c in set(classes):
            at = torch.tensor([i for i in range(b) if slices[i] == c], device=DEV)
            assert err(got[:, at], ref[:, at]) <= 16 * m * (
                (2 * n) ** 0.5 * 2.0 ** -(48 if c == 7 else 30) + 8 * U + (2 * n) ** 0.5 * U)
    assert len(ways) > 1  # more launches where moduli or columns take turns
    # one modulus of H does not fit: an error, not a result, and the next call works
    with limit(2 * MB), pytest.raises(chase.ChaseError) as e:
        chase.chase_filter_mixed(h, v.clone(), [m] * b, slices, 1.6, -1.5, -0.9)
    assert e.value.status == chase.CHASE_OUT_OF_MEMORY
    chase.chase_filter_mixed(h, v.clone(), [m] * b, slices, 1.6, -1.5, -0.9)


@pytest.mark.parametrize("mb", [4, 16, 20, 40, 0])
def test_residuals_and_rayleigh_ritz(mb):
    n, b = 1200, 40
    h = hermitian(n, 5, False)
    q = torch.linalg.qr(gauss(n, b, 6, False))[0].t().contiguous().t()
    lam = np.linspace(-1.0, 1.0, b)
    want = torch.linalg.norm(h @ q - q * torch.from_numpy(lam).to(DEV), dim=0).cpu().numpy()
    with limit(mb * MB):
        assert np.max(np.abs(chase.chase_residuals(h, q, lam) - want)) <= 20 * n ** 0.5 * U
    g = q.conj().t() @ (h @ q)
    theta = torch.linalg.eigvalsh(0.5 * (g + g.conj().t())).cpu().numpy()
    x = q.clone()
    with limit(max(mb, 8) * MB if mb else 0):
        ritz, resid = chase.chase_rayleigh_ritz(h, x)
    assert np.max(np.abs(ritz - theta)) <= 20 * (b + n ** 0.5) * U
    assert float(torch.linalg.norm(x.conj().t() @ x - torch.eye(b, device=DEV))) <= 20 * (b + n ** 0.5) * U
    r = torch.linalg.norm(h @ x - x * torch.from_numpy(ritz).to(DEV), dim=0).cpu().numpy()
    assert np.max(np.abs(resid - r)) <= 50 * (b + n ** 0.5) * U


SOLVES = [(p, mb) for p in (chase.CHASE_FP64, chase.CHASE_SPLIT_BF16, chase.CHASE_SPLIT_BF16_RR,
                            chase.CHASE_SPLIT_BF16_ADAPT) for mb in (18, 24, 40, 0)] + [(chase.CHASE_FP64, 12)]


@pytest.mark.parametrize("precision,mb", SOLVES)
def test_solve(precision, mb):
    n, nev, nex = 1200, 24, 16
    lam = synth.spectrum_uniform(n, 7, device=DEV)
    h = synth.hermitian_dft(lam, 8)
    v = synth.gaussian_block(n, nev + nex, 9, device=DEV)
    s = synth.gaussian_block(n, 5, 10, device=DEV)
    with limit(mb * MB):
        st, ritz, _, _ = chase.chase_solve(h, nev, nex, 1e-10, v, s,
                                           opts=chase.chase_opts_default(precision=precision))
    assert st == chase.CHASE_OK
    assert np.max(np.abs(ritz[:nev] - lam.cpu().numpy()[:nev])) <= 1e-10 * float(lam.abs().max())


@pytest.mark.parametrize("mb", [12, 24, 0])
def test_single_precision_solve(mb):
    n, nev, nex = 1200, 24, 16
    lam = synth.spectrum_uniform(n, 11, device=DEV)
    h = synth.hermitian_dft(lam, 12).to(torch.complex64)
    v = synth.gaussian_block(n, nev + nex, 13, device=DEV).to(torch.complex64)
    s = synth.gaussian_block(n, 5, 14, device=DEV).to(torch.complex64)
    with limit(mb * MB):
        st, ritz, _, _ = chase.chase_solve_c32(h, nev, nex, 1e-5, v, s)
    assert st == chase.CHASE_OK
    assert np.max(np.abs(ritz[:nev] - lam.cpu().numpy()[:nev])) <= 1e-5 * float(lam.abs().max())


SHAPES = [(500, 30), (300, 20), (257, 9), (300, 40), (129, 12), (400, 24)]


# H of the batch: 13 MB; its planes 27 to 53 MB, of the blocks 9 MB
@pytest.mark.parametrize("split", [False, True])
def test_batched_filter(split):
    m = 6
    hs = [hermitian(n, 20 + i, False) for i, (n, b) in enumerate(SHAPES)]
    vs = [gauss(n, b, 30 + i, False) for i, (n, b) in enumerate(SHAPES)]
    refs = [reference(h, v, m, 1.6, -1.5, -0.9) for h, v in zip(hs, vs)]
    ways = set()
    for mb in (4, 6, 12, 24, 48, 0):
        got = [v.clone() for v in vs]
        with limit(mb * MB):
            st = chase.chase_filter_batched(hs, got, [np.full(b, m, dtype=np.int32) for _, b in SHAPES],
                                            [1.6] * 6, [-1.5] * 6, [-0.9] * 6,
                                            precision=chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64)
        ways.add((st["launches"], st["tile_config"] < 0))
        assert st["matvecs"] == m * sum(b for _, b in SHAPES)
        for (n, b), v, ref in zip(SHAPES, got, refs):
            assert err(v, ref) <= bar(n, m, "c128", split)
    assert len({k for k, rns in ways if rns}) > 1  # the batch at once, and in parts
    assert not all(rns for _, rns in ways)  # and FP64 tiles for what does not fit alone


@pytest.mark.parametrize("precision", [chase.CHASE_FP64, chase.CHASE_SPLIT_BF16, chase.CHASE_SPLIT_BF16_RR])
@pytest.mark.parametrize("mb", [48, 160, 0])
def test_batched_solve(precision, mb):
    shapes = [(500, 20, 10), (300, 12, 6), (400, 16, 8)]
    lam = [synth.spectrum_uniform(n, 40 + n, device=DEV) for n, _, _ in shapes]
    hs = [synth.hermitian_dft(x, 41) for x in lam]
    vs = [synth.gaussian_block(n, nev + nex, 42, device=DEV) for n, nev, nex in shapes]
    ss = [synth.gaussian_block(n, 5, 43, device=DEV) for n, _, _ in shapes]
    with limit(mb * MB):
        out = chase.chase_solve_batched(hs, [s[1] for s in shapes], [s[2] for s in shapes], [1e-10] * 3, vs, ss,
                                        opts=chase.chase_opts_default(precision=precision))
    assert out[0] == chase.CHASE_OK
    for x, ritz, (n, nev, nex) in zip(lam, out[2], shapes):
        assert np.max(np.abs(ritz[:nev] - x.cpu().numpy()[:nev])) <= 1e-10 * float(x.abs().max())
