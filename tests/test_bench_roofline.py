"""The roofline bench.py reports for the flux launch, on the CPU."""
import pytest

import bench

FP64 = {"sustained_tflops": 1.252, "burst_tflops": 1.254}


def test_flux_roofline_is_a_share_of_what_bounds_the_launch():
    """Shares of peaks stay below one, also at a launch time at which the method's FP64 work
    would exceed the FP64 peak; that work is named apart."""
    n = 256 ** 3
    slow, fast = (bench.flux_roofline(t, n, 152, 2070.0, FP64) for t in (10.76e-3, 7.3e-3))
    for r, t in ((slow, 10.76e-3), (fast, 7.3e-3)):
        assert 0.0 < r["frac"] < 1.0 and r["frac"] == pytest.approx(r["achieved"] / r["peak"])
        assert 0.0 < r["executed_fp64"]["frac"] < 1.0
        assert r["peak"] == pytest.approx(4 * 152 * 2.07)
        assert r["equivalent_fp64"]["tflops"] == pytest.approx(254.4 * 3 * n / t / 1e12)
    assert fast["equivalent_fp64"]["over_peak"] > 1.0
    assert fast["achieved"] / slow["achieved"] == pytest.approx(10.76 / 7.3)


def test_flux_roofline_takes_fewer_fp64_operations_than_the_method_has():
    assert bench.FLUX_FP64_FLOP_PER_CELL < 0.5 * 3 * bench.FLUX_FLOPS_PER_CELL_DIR
    assert bench.FLUX_TRAFFIC_BYTES_PER_CELL > bench.FLUX_BYTES_PER_CELL
