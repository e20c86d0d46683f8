"""The benchmark's line on lattice totals: achieved, peak, unit and fraction
are those of the bound that it names."""
import pytest

import bench


@pytest.mark.parametrize("prec,bytes_per_site", [("fp32_shifted", 152), ("fp64", 304)])
def test_fraction_is_of_the_named_bound(prec, bytes_per_site):
    n, t, peak, tflops = 256 ** 3, 0.5e-3, 6800.0, 1.05
    roof = bench._reduce_line(prec, t, n, tflops, peak, "measured")["roofline"]
    gbs = bytes_per_site * n / t / 1e9
    assert roof["hbm_frac"] == pytest.approx(gbs / peak)
    if prec == "fp32_shifted":
        assert (roof["bound"], roof["unit"], roof["peak"]) == ("hbm", "GB/s", peak)
        assert roof["achieved"] == pytest.approx(gbs) and roof["frac"] == roof["hbm_frac"]
    else:
        assert roof["bound"] == "alu (FP64 pipe)" and roof["peak"] == tflops / 2
        assert roof["frac"] == pytest.approx(roof["fp64_adds_per_site"] * n / t / 1e12 / (tflops / 2))
