"""Batches on both sides of the rule that chooses between residue products and
FP64 tiles (many problems of few rows take the FP64 tiles, in either precision),
and products whose tiles each pair of blocks takes one after the other (all
problems up to N = 256) or in turn, with one large problem among small ones.

Tolerance: as in test_gpu_scales.py."""

import numpy as np
import pytest
import torch

from paper_1805_10121_gb300 import chase, synth
from tests.test_gpu_rns import gauss, hermitian, reference
from tests.test_gpu_scales import bar, err

pytestmark = pytest.mark.gpu

TINY = [(16, 4)] * 60 + [(40, 9)] * 200
SMALL = [(256, 19), (129, 7), (200, 33), (64, 5), (255, 1), (130, 40)] * 3


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


@pytest.mark.parametrize("shapes,rns", [(TINY, False), (SMALL, True), (SMALL + [(257, 12)], True),
                                        (TINY + [(700, 40)], True)])
@pytest.mark.parametrize("split", [False, True])
def test_batch(shapes, rns, split):
    # degrees that retire columns, so that later steps hold fewer tiles; of many
    # equal shapes only five problems differ
    made = {}
    for i, (n, b) in enumerate(shapes):
        if (n, b, i % 5) not in made:
            h, v = hermitian(n, i, False), gauss(n, b, 100 + i, False)
            made[n, b, i % 5] = h, v, [reference(h, v, m, 1.6, -1.5, -0.9) for m in (2, 4, 6)]
    hs, vs, refs = zip(*(made[n, b, i % 5] for i, (n, b) in enumerate(shapes)))
    vs = [v.clone() for v in vs]
    degs = [2 * (1 + np.arange(b, dtype=np.int32) % 3) for n, b in shapes]
    st = chase.chase_filter_batched(hs, vs, degs, [1.6] * len(hs), [-1.5] * len(hs), [-0.9] * len(hs),
                                    precision=chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64)
    assert (st["tile_config"] < 0) == rns
    for (n, b), v, ref in zip(shapes, vs, refs):
        for k in range(min(3, b)):
            assert err(v[:, k::3], ref[k][:, k::3]) <= bar(max(n, 64), 2 * (k + 1), split)


@pytest.mark.parametrize("precision", [chase.CHASE_FP64, chase.CHASE_SPLIT_BF16])
def test_solve_with_more_problems_than_streams(precision):
    # problems of different sizes follow one another on each stream
    shapes = [(130 + 37 * ((7 * i) % 20), 6 + i % 9, 3 + i % 4) for i in range(36)]
    lam = [synth.spectrum_uniform(n, 50 + i, device="cuda") for i, (n, _, _) in enumerate(shapes)]
    hs = [synth.hermitian_dft(x, 51 + i) for i, x in enumerate(lam)]
    vs = [synth.gaussian_block(n, a + x, 52 + i, device="cuda") for i, (n, a, x) in enumerate(shapes)]
    ss = [synth.gaussian_block(n, 5, 53 + i, device="cuda") for i, (n, _, _) in enumerate(shapes)]
    out = chase.chase_solve_batched(hs, [s[1] for s in shapes], [s[2] for s in shapes], 1e-10, vs, ss,
                                    opts=chase.chase_opts_default(precision=precision))
    assert out[0] == chase.CHASE_OK
    for h, v, x, ritz, (n, nev, nex) in zip(hs, vs, lam, out[2], shapes):
        top = float(x.abs().max())
        assert np.max(np.abs(ritz[:nev] - x.cpu().numpy()[:nev])) <= 1e-10 * top
        y = v[:, :nev]
        r = torch.linalg.norm(h @ y - y * torch.from_numpy(ritz[:nev]).to(y.device), dim=0)
        assert float(r.max()) <= 1.05e-10 * top
