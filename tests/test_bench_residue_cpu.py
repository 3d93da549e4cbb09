"""bench.py's rooflines of the residue products on synthetic per-solve
statistics: fractions follow from the planes executed, the time and the measured
BF16 peak, per precision.  CPU only."""

import pytest

import bench

PK = {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0}
KEYS = {"bound", "kernel", "achieved", "peak", "unit", "frac", "traffic"}


def stats(**kw):
    return {"flops_filter": 0.0, "t_filter": 0.0, "flops_rr_product": 0.0, "t_rr_product": 0.0,
            "lanczos_matvecs": 0, "t_lanczos": 0.0, **kw}


@pytest.mark.parametrize("precision,n,filt,rr", [
    ("fp64", 8000, 14, 14), ("split", 8000, 11, 14), ("split", 40000, 12, 14), ("split_adapt", 8000, 11, 14),
    ("split_rr", 8000, 12, 12)])
def test_solve(precision, n, filt, rr):
    s = [stats(flops_filter=1.0e14, t_filter=1.0, flops_rr_product=4.0e13, t_rr_product=0.5)] * 2
    main, other = bench.residue_roofline(s, n, PK, "measured", precision)
    assert KEYS <= set(main) and KEYS <= set(other)
    assert "the filter steps" in main["kernel"] and "Rayleigh-Ritz" in other["kernel"]
    assert main["fp64_equivalent_tflops"] == pytest.approx(100.0)
    assert main["achieved"] == pytest.approx(0.5 * filt * 100.0)
    assert main["frac"] == pytest.approx(0.5 * filt * 100.0 / 1700.0, rel=1e-3)
    assert other["achieved"] == pytest.approx(0.5 * rr * 80.0)


def test_the_longer_phase_comes_first():
    s = [stats(flops_filter=1.0e13, t_filter=0.1, flops_rr_product=1.0e13, t_rr_product=0.2)]
    main, other = bench.residue_roofline(s, 8000, PK, "measured", "split")
    assert "Rayleigh-Ritz" in main["kernel"] and "filter" in other["kernel"]
    main, _ = bench.residue_roofline([stats()], 8000, PK, "measured", "fp64")  # nothing timed
    assert main["achieved"] == 0.0 and main["frac"] == 0.0


def test_lanczos_on_planes():
    n = 8000
    e = bench.lanczos_entry([stats(lanczos_matvecs=25, t_lanczos=0.0142)], n, PK, "measured", planes=True)
    gbs = 28.0 * n * n * 25 / 0.0142 / 1e9
    assert e["achieved"] == pytest.approx(gbs, rel=1e-3) and e["frac"] == pytest.approx(gbs / 6800.0, rel=1e-3)
    assert e["bound"] == "hbm" and "rns_gemm_kernel" in e["kernel"]


def test_residue_bytes_per_product():
    # 11 planes of H (one per modulus), 22 of the block, residues of 22 planes
    n, b = 8000, 480
    assert bench.residue_algorithmic_bytes(n, b) == pytest.approx(
        11 * 2 * n * n + 22 * 2 * n * b + 22 * 2 * n * b)
