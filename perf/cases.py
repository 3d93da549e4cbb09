"""Performance cases: the calls a user of this library makes, over the sizes they make them at.

A case names one call of the public Python binding with its sizes; prepare()
builds the device arrays a calling program has in hand, run() makes the call,
work() counts what it cannot do without, and exact() gives its result in
64-bit arithmetic from plain torch operations.

Sizes: the single problem N = 1000 (nev 50, nex 20), the batch of problems
with N in [256, 2048] (nev 5 %, nex 2 % of N), the N = 8000 sequence, and the
served sequences N in {2048 ... 16384} (nev 4 % of N, nex 20 % of nev), with
odd sizes between them.  Blocks are filtered with one degree for every column
(the first filter of a solve: 20) or with a degree per column (later ones: 8
to 36, any order).  Solves start cold from random vectors, or warm from the
vectors of the problem before in a sequence; the split filter runs with the
degree cap 64 and 6 extra degrees that the benchmark gives it.
"""

import math

import numpy as np
import torch

from paper_1805_10121_gb300 import chase

DEVICE = "cuda"
FP64, SPLIT = chase.CHASE_FP64, chase.CHASE_SPLIT_BF16
_PRECISION = {"fp64": FP64, "split": SPLIT, "adapt": chase.CHASE_SPLIT_BF16_ADAPT}


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest problem of a batch, filtered on its own: launches and host work count
        {"name": "filter_fp64_n256", "kind": "filter", "field": "c128", "split": False, "n": 256, "b": 19,
         "deg": 0, "spectrum": "uniform"},
        # a later filter of the single problem N = 1000, every column with its own degree
        {"name": "filter_fp64_n1000", "kind": "filter", "field": "c128", "split": False, "n": 1000, "b": 70,
         "deg": 0, "spectrum": "clustered"},
        # the first filter of a served N = 4096 problem in plain FP64
        {"name": "filter_fp64_n4096", "kind": "filter", "field": "c128", "split": False, "n": 4096, "b": 197,
         "deg": 20, "spectrum": "dft"},
        # a real symmetric problem of odd size in FP64
        {"name": "filter_real_n2501", "kind": "filter", "field": "f64", "split": False, "n": 2501, "b": 151,
         "deg": 0, "spectrum": "dft"},
        # the single-precision solver's filter
        {"name": "filter_c32_n2000", "kind": "filter", "field": "c64", "split": False, "n": 2000, "b": 140,
         "deg": 0, "spectrum": "dft"},
        # a later filter of the smallest served problem on the split product
        {"name": "filter_split_n2048", "kind": "filter", "field": "c128", "split": True, "n": 2048, "b": 99,
         "deg": 0, "spectrum": "dft"},
        # the first filter of the largest served problem on the split product
        {"name": "filter_split_n16384", "kind": "filter", "field": "c128", "split": True, "n": 16384, "b": 788,
         "deg": 20, "spectrum": "dft"},
        # many independent problems of uneven size in one call
        {"name": "filter_batched_split_32", "kind": "batched", "split": True, "p": 32, "lo": 256, "hi": 2048,
         "deg": 0, "spectrum": "uniform"},
        # the orthogonalisation inside an iteration of the N = 8000 sequence: part of the block is locked
        {"name": "orthonormalize_n8000", "kind": "orth", "n": 8000, "nconv": 180, "b": 300},
        # Rayleigh-Ritz with residuals of a served N = 4096 problem
        {"name": "rayleigh_ritz_n4096", "kind": "rr", "n": 4096, "b": 197, "spectrum": "dft"},
        # a whole cold solve of the single problem N = 1000 in plain FP64
        {"name": "solve_fp64_n1000", "kind": "solve", "precision": "fp64", "warm": False, "n": 1000, "nev": 50,
         "nex": 20, "spectrum": "clustered"},
        # a whole solve inside a sequence: warm-started from the previous problem's vectors, split filter
        {"name": "solve_split_warm_n4095", "kind": "solve", "precision": "split", "warm": True, "n": 4095,
         "nev": 164, "nex": 33, "spectrum": "dft"},
    ]


def draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return max(lo, min(hi, n))

    def block(n, most):
        return max(8, min(int(n * rng.uniform(0.03, 0.09)) + 1, int(most), n // 2))

    kind = rng.choice(["filter", "filter", "filter", "filter", "batched", "orth", "rr", "solve"])
    deg = rng.choice([0, 0, 20])
    if kind == "filter":
        field = rng.choice(["c128", "c128", "f64", "c64", "f32"])
        split = field in ("c128", "f64") and rng.random() < 0.6
        n = size(256, 12000 if split else 4000 if field in ("c128", "f64") else 2400)
        # flops as the listed FP64 and split filters have at most
        per = (8.0 if field in ("c128", "c64") else 2.0) * n * n * 20
        return {"kind": kind, "field": field, "split": split, "n": n,
                "b": block(n, (3.0e13 if split else 4.5e11) / per), "deg": deg,
                "spectrum": rng.choice(["uniform", "dft"])}
    if kind == "batched":
        split = rng.random() < 0.7
        return {"kind": kind, "split": split, "p": rng.randint(3, 32 if split else 12), "lo": 256,
                "hi": size(600, 2048), "deg": deg, "spectrum": "uniform"}
    if kind == "orth":
        n = size(400, 8000)
        b = block(n, 300)
        return {"kind": kind, "n": n, "nconv": rng.choice([0, b // 3, b]), "b": b}
    if kind == "rr":
        n = size(300, 5000)
        return {"kind": kind, "n": n, "b": block(n, 240), "spectrum": rng.choice(["uniform", "dft"])}
    precision = rng.choice(["fp64", "split", "adapt"])
    warm = rng.random() < 0.5
    n = size(300, 1000 if precision == "fp64" else 4000)
    nev = max(4, int(0.04 * n))
    return {"kind": "solve", "precision": precision, "warm": warm, "n": n, "nev": nev,
            "nex": max(3, int(0.3 * nev)), "spectrum": rng.choice(["clustered", "dft"])}


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    return g


def _spectrum(kind, n, g):
    """Ascending eigenvalues: uniform in [-1, 1]; a cluster of 6 % in [-1, -0.9] below the rest; or the DFT-like
    law, a dense band in [-2, 0] (a quarter of the values) below a sparse tail up to 50."""
    u = torch.rand(n, dtype=torch.float64, device=DEVICE, generator=g)
    if kind == "uniform":
        lam = -1.0 + 2.0 * u
    elif kind == "clustered":
        m = max(1, (6 * n) // 100)
        lam = torch.cat([-1.0 + 0.1 * u[:m], -0.9 + 1.9 * (1.0 - u[m:])])
    else:
        m = n // 4
        lam = torch.cat([-2.0 + 2.0 * u[:m], 50.0 * (1.0 - u[m:]) ** 2])
    return torch.sort(lam).values


class _Basis:
    """The eigenvectors of a test matrix: the dense unitary D1 F D2 F D3 with the unitary DFT F and random phase
    diagonals, or, real, D1 C D2 C D3 with the Hartley transform C and random signs."""

    def __init__(self, n, real, g):
        self.real = real
        r = torch.rand(3, n, dtype=torch.float64, device=DEVICE, generator=g)
        self.d = torch.where(r < 0.5, -1.0, 1.0).to(torch.float64) if real else torch.polar(
            torch.ones_like(r), 2.0 * math.pi * r)

    def _t(self, x, inverse):
        if not self.real:
            return (torch.fft.ifft if inverse else torch.fft.fft)(x, dim=0, norm="ortho")
        y = torch.fft.fft(x.to(torch.complex128), dim=0, norm="ortho")
        return y.real - y.imag  # Hartley: its own inverse

    def mul(self, x):
        x = self._t(self.d[2][:, None] * x, False)
        return self.d[0][:, None] * self._t(self.d[1][:, None] * x, False)

    def adj(self, x):
        x = self._t(self.d[0].conj()[:, None] * x, True)
        return self.d[2].conj()[:, None] * self._t(self.d[1].conj()[:, None] * x, True)


def _columns(x):
    """The same matrix with contiguous columns, as the library takes it."""
    return x.t().contiguous().t()


def _matrix(n, spectrum, real, g, chunk=2048):
    lam = _spectrum(spectrum, n, g)
    q = _Basis(n, real, g)
    dt = torch.float64 if real else torch.complex128
    h = torch.empty(n, n, dtype=dt, device=DEVICE).t()
    for j0 in range(0, n, chunk):
        j1 = min(n, j0 + chunk)
        e = torch.zeros(n, j1 - j0, dtype=dt, device=DEVICE)
        e[torch.arange(j0, j1, device=DEVICE), torch.arange(j1 - j0, device=DEVICE)] = 1.0
        h[:, j0:j1] = q.mul(lam[:, None] * q.adj(e))
    for i0 in range(0, n, chunk):  # the Hermitian part, block pair by block pair
        for j0 in range(i0, n, chunk):
            s, t = slice(i0, i0 + chunk), slice(j0, j0 + chunk)
            a = 0.5 * (h[s, t] + h[t, s].conj().t())
            h[s, t] = a
            h[t, s] = a.conj().t()
    return h, lam, q


def _gauss(n, b, real, g):
    if real:
        return torch.randn(b, n, dtype=torch.float64, device=DEVICE, generator=g).t()
    x = torch.randn(b, n, 2, dtype=torch.float64, device=DEVICE, generator=g)
    return torch.view_as_complex(x).mul_(1.0 / math.sqrt(2.0)).t()


def _degrees(deg, b, seed):
    if deg:
        return np.full(b, deg, dtype=np.int32)
    return (2 * np.random.RandomState(seed % (1 << 31)).randint(4, 19, b)).astype(np.int32)


_TYPES = {"c128": torch.complex128, "f64": torch.float64, "c64": torch.complex64, "f32": torch.float32}


def _filter_inputs(n, b, deg, spectrum, field, g, seed):
    real = field in ("f64", "f32")
    h, lam, _ = _matrix(n, spectrum, real, g)
    v = _gauss(n, b, real, g)
    top = max(abs(float(lam[0])), abs(float(lam[-1])))
    return {"H": h.to(_TYPES[field]), "V": v.to(_TYPES[field]), "deg": _degrees(deg, b, seed),
            "b_sup": float(lam[-1]) + 0.01 * top, "mu1": float(lam[0]), "mu_nn": float(lam[b])}


def _near(q, n, b, g):
    """The b lowest eigenvectors of the matrix with basis q, each about 2 % off."""
    e = 0.02 / math.sqrt(n) * _gauss(n, b, False, g)
    e[torch.arange(b, device=DEVICE), torch.arange(b, device=DEVICE)] += 1.0
    return q.mul(e)


def _batch_sizes(case):
    """Sizes over the whole range in no particular order, odd ones among them."""
    r = np.random.RandomState(case["p"])
    n = np.linspace(case["lo"], case["hi"], case["p"]).round().astype(int)
    n = [min(int(v) | 1 if i % 2 else int(v), case["hi"]) for i, v in enumerate(n)]
    return [(n[i], math.ceil(0.05 * n[i]) + math.ceil(0.02 * n[i])) for i in r.permutation(case["p"])]


def prepare(case, seed):
    g = _gen(seed)
    k = case["kind"]
    if k == "filter":
        return dict(_filter_inputs(case["n"], case["b"], case["deg"], case["spectrum"], case["field"], g, seed),
                    case=case)
    if k == "batched":
        one = [_filter_inputs(n, b, case["deg"], case["spectrum"], "c128", g, seed + 31 * i)
               for i, (n, b) in enumerate(_batch_sizes(case))]
        return {"case": case, "problems": one}
    if k == "orth":
        # a filtered block: columns of very different sizes along the wanted directions, condition about 1e3,
        # beside locked vectors that it still has components of
        n, b, m = case["n"], case["b"], case["nconv"]
        q = _Basis(n, False, g)
        e = torch.zeros(n, max(m, 1), dtype=torch.complex128, device=DEVICE)
        e[torch.arange(max(m, 1), device=DEVICE), torch.arange(max(m, 1), device=DEVICE)] = 1.0
        y = _columns(q.mul(e))[:, :m]
        w = torch.linalg.qr(_gauss(b, b, False, g))[0]
        s = torch.logspace(0.0, -3.0, b, dtype=torch.float64, device=DEVICE)
        v = (_gauss(n, b, False, g) * s[None, :]) @ w
        if m:
            v = v + 0.5 * y @ _gauss(m, b, False, g)
        return {"case": case, "Y": y, "V": _columns(v)}
    if k == "rr":
        # an orthonormal block near the lowest eigenvectors, as it comes out of the orthogonalisation
        n, b = case["n"], case["b"]
        h, lam, q = _matrix(n, case["spectrum"], False, g)
        x = torch.linalg.qr(_near(q, n, b, g) @ torch.linalg.qr(_gauss(b, b, False, g))[0])[0]
        return {"case": case, "H": h, "Q": _columns(x)}
    n, nx = case["n"], case["nev"] + case["nex"]
    h, lam, q = _matrix(n, case["spectrum"], False, g)
    s = {"case": case, "H": h, "V": _gauss(n, nx, False, g), "Lambda": None, "starts": _gauss(n, 5, False, g)}
    more = {} if case["precision"] == "fp64" else {"deg_extra": 6, "deg_max": 64}
    if case["warm"]:
        # the vectors and values of the problem before this one in a sequence
        s["V"] = _columns(torch.linalg.qr(_near(q, n, nx, g))[0])
        s["Lambda"] = (lam[:nx] + 1e-3 * torch.randn(nx, dtype=torch.float64, device=DEVICE, generator=g)).cpu().numpy()
        s["starts"] = s["starts"][:, :1]
        more["approx"] = 1
    s["opts"] = chase.chase_opts_default(precision=_PRECISION[case["precision"]], **more)
    return s


# ---------------------------------------------------------------- one pass

_FILTER = {"c128": chase.chase_filter, "f64": chase.chase_filter_real, "c64": chase.chase_filter_c32,
           "f32": chase.chase_filter_f32}


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "filter":
        v = s["V"].clone()  # the library filters in place
        more = {"precision": SPLIT if case["split"] else FP64} if case["field"] in ("c128", "f64") else {}
        return _FILTER[case["field"]](s["H"], v, s["deg"], s["b_sup"], s["mu1"], s["mu_nn"], **more)
    if k == "batched":
        p = s["problems"]
        v = [x["V"].clone() for x in p]
        chase.chase_filter_batched([x["H"] for x in p], v, [x["deg"] for x in p], [x["b_sup"] for x in p],
                                   [x["mu1"] for x in p], [x["mu_nn"] for x in p],
                                   precision=SPLIT if case["split"] else FP64)
        return v
    if k == "orth":
        return chase.chase_orthonormalize(s["Y"], s["V"].clone())
    if k == "rr":
        q = s["Q"].clone()
        ritz, resid = chase.chase_rayleigh_ritz(s["H"], q)
        # Ritz vectors are defined up to a phase: the first entry real and positive
        return {"ritz": ritz, "resid": resid, "Q": q * (q[:1].conj() / q[:1].abs())}
    # of a solve, the nev converged eigenvalues are determined by H; its vectors and residuals only to the
    # tolerance that it was asked for
    st, lam, _, _ = chase.chase_solve(s["H"], case["nev"], case["nex"], 1e-10, s["V"].clone(), s["starts"],
                                      Lambda=s["Lambda"], opts=s["opts"])
    return {"status": st, "Lambda": lam[:case["nev"]]}


# ---------------------------------------------------------------- what a pass cannot do without

_MEAN_DEGREE = 22.0


def work(case):
    k = case["kind"]
    if k == "filter":
        size = {"c128": 16, "f64": 8, "c64": 8, "f32": 4}[case["field"]]
        mv = 8.0 if case["field"] in ("c128", "c64") else 2.0
        n, b = case["n"], case["b"]
        return {"bytes": size * (n * n + 2.0 * n * b), "flops": mv * n * n * b * (case["deg"] or _MEAN_DEGREE)}
    if k == "batched":
        z = _batch_sizes(case)
        return {"bytes": sum(16.0 * (n * n + 2 * n * b) for n, b in z),
                "flops": sum(8.0 * n * n * b * (case["deg"] or _MEAN_DEGREE) for n, b in z)}
    if k == "orth":
        n, b, m = case["n"], case["b"], case["nconv"]
        # Q of [Y V] keeping Y: the projection (two products) and a Householder-like QR of V
        return {"bytes": 16.0 * n * (m + 2 * b), "flops": 16.0 * n * m * b + 8.0 * n * b * b}
    if k == "rr":
        n, b = case["n"], case["b"]
        return {"bytes": 16.0 * (n * n + 2 * n * b), "flops": 8.0 * n * n * b + 20.0 * n * b * b}
    n, b = case["n"], case["nev"] + case["nex"]
    # about four filters of the block, each with one Rayleigh-Ritz and orthogonalisation
    return {"bytes": 16.0 * (n * n + 2 * n * b), "flops": 4 * (8.0 * n * n * b * (_MEAN_DEGREE + 1) + 28.0 * n * b * b)}


# ---------------------------------------------------------------- the same in plain 64-bit torch

def _exact_filter(h, v, deg, b_sup, mu1, mu_nn):
    up = torch.complex128 if v.is_complex() else torch.float64
    h, x = h.to(up), v.to(up)
    c, e = 0.5 * (b_sup + mu_nn), 0.5 * (b_sup - mu_nn)
    s1 = e / (mu1 - c)
    d = torch.as_tensor(np.asarray(deg), device=x.device)
    out = x.clone()
    prev, cur = x, (s1 / e) * (h @ x - c * x)
    sigma = s1
    for i in range(2, int(d.max()) + 1):
        tau = 1.0 / (2.0 / s1 - sigma)
        prev, cur = cur, (2.0 * tau / e) * (h @ cur - c * cur) - (tau * sigma) * prev
        sigma = tau
        out = torch.where((d == i)[None, :], cur, out)
    return out


def exact(case, seed):
    k = case["kind"]
    if k not in ("solve", "orth", "rr") and work(case)["flops"] > 6e12:
        return None  # over a few seconds of 64-bit products
    s = prepare(case, seed)
    if k == "filter":
        return _exact_filter(s["H"], s["V"], s["deg"], s["b_sup"], s["mu1"], s["mu_nn"])
    if k == "batched":
        return [_exact_filter(x["H"], x["V"], x["deg"], x["b_sup"], x["mu1"], x["mu_nn"]) for x in s["problems"]]
    if k == "orth":
        v, y = s["V"], s["Y"]
        for _ in range(2):
            v = v - y @ (y.conj().t() @ v)
        q, r = torch.linalg.qr(v)
        d = torch.diagonal(r)
        return q * (d / d.abs())[None, :]
    if k == "rr":
        h, q = s["H"], s["Q"]
        hq = h @ q
        g = q.conj().t() @ hq
        lam, w = torch.linalg.eigh(0.5 * (g + g.conj().t()))
        x, hx = q @ w, hq @ w
        return {"ritz": lam, "resid": torch.linalg.vector_norm(hx - x * lam[None, :], dim=0),
                "Q": x * (x[:1].conj() / x[:1].abs())}
    lam = torch.linalg.eigvalsh(s["H"])
    return {"status": None, "Lambda": lam[:case["nev"]]}
