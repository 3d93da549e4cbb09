"""Filters whose degree steps are chained (reconstruction and slicing for the
next step in one kernel, a cluster per column): columns that retire at every
step, sizes at the edges of a thread's two rows, a block's 256 or 512 and the
largest N that is chained, all four types, and columns whose squares leave
FP32's range beside a zero column.

Tolerance: as in test_gpu_rns.py (operands rounded to 2^-L of a norm and FP64
roundings, or FP32 storage, for each of the m products of a filter whose
values stay within 2 m of the input's norm)."""

import numpy as np
import pytest
import torch

from paper_1805_10121_gb300 import chase
from tests.test_gpu_rns import DEV, U, gauss, hermitian, reference

pytestmark = pytest.mark.gpu

FILTER = {"c128": chase.chase_filter, "f64": chase.chase_filter_real, "c64": chase.chase_filter_c32,
          "f32": chase.chase_filter_f32}
TYPE = {"c128": torch.complex128, "f64": torch.float64, "c64": torch.complex64, "f32": torch.float32}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


def bar(n, m, field, split):
    unit = 2.0 ** -24 if field in ("c64", "f32") else U
    bits = 30 if field in ("c64", "f32") else 48 if split else 60
    return 16 * m * ((2 * n) ** 0.5 * 2.0 ** -bits + 8 * unit + (2 * n) ** 0.5 * U)


@pytest.mark.parametrize("n,b", [(128, 7), (255, 12), (256, 30), (257, 19), (513, 40), (1025, 25), (2047, 33),
                                 (2049, 21), (4095, 9), (4096, 17), (4097, 17)])
@pytest.mark.parametrize("field,split", [("c128", False), ("c128", True), ("f64", False), ("f64", True),
                                         ("c64", False), ("f32", False)])
def test_every_column_its_degree(n, b, field, split):
    real = field in ("f64", "f32")
    h, v = (x.to(TYPE[field]).t().contiguous().t() for x in (hermitian(n, n, real), gauss(n, b, b, real)))
    deg = 2 * np.random.RandomState(n + b).randint(1, 6, b)
    up = torch.float64 if real else torch.complex128
    got = v.clone()
    more = {"precision": chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64} if field in ("c128", "f64") else {}
    FILTER[field](h, got, deg.astype(np.int32), 1.6, -1.5, -0.9, **more)
    for m in sorted(set(deg)):
        at = torch.from_numpy(np.flatnonzero(deg == m)).to(DEV)
        ref = reference(h.to(up), v[:, at].to(up), int(m), 1.6, -1.5, -0.9)
        e = torch.linalg.norm(got[:, at].to(up) - ref, dim=0) / torch.linalg.norm(ref, dim=0)
        assert float(e.max()) <= bar(n, int(m), field, split)


@pytest.mark.parametrize("n", [300, 1025, 3000])
@pytest.mark.parametrize("split", [False, True])
def test_columns_of_extreme_scale(n, split):
    h, v, m = hermitian(n, 5, False), gauss(n, 16, 6, False), 6
    f = torch.ones(16, dtype=torch.float64, device=DEV)
    f[1::5], f[2::5], f[3::5], f[4] = 1e-140, 1e-13, 1e30, 0.0
    ref = reference(h, v, m, 1.6, -1.5, -0.9)
    got = (v * f[None, :]).t().contiguous().t()
    chase.chase_filter(h, got, [m] * 16, 1.6, -1.5, -0.9,
                       precision=chase.CHASE_SPLIT_BF16 if split else chase.CHASE_FP64)
    assert float(got[:, 4].abs().max()) == 0.0
    keep = torch.arange(16, device=DEV) != 4
    d = got[:, keep] / f[None, keep] - ref[:, keep]
    e = torch.linalg.norm(d, dim=0) / torch.linalg.norm(ref[:, keep], dim=0)
    assert float(e.max()) <= bar(n, m, "c128", split)
