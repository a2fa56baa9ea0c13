"""CPU checks of the fixed-point figures beside bench.py's roofline: the multiply-adds a transform issues follow from the
radices of its plan, and the peak is the rate of the multiply pipe over them."""
import math

import pytest


# 6: one stage; 18 = 3 x 6; 96 = 4 x 2 x 12; 768 = 4 x 4 x 4 x 12; 864 = 4 x 2 x 3 x 3 x 12
@pytest.mark.parametrize("n,madds", [(6, 2.0), (12, 2.0), (18, 2 + 10 + 2), (96, 0 + 6 + 11 + 2), (768, 9 + 9 + 11 + 2),
                                     (864, 6 + 10 + 10 + 11 + 2)])
def test_multiply_adds_per_point(n, madds):
    import bench
    assert bench.fixed_point_madds(n) == pytest.approx(madds)


@pytest.mark.parametrize("kernel,n", [("fft_x_inverse", 768), ("fft_z_forward", 96)])
def test_peak_uses_the_length_of_the_pass(kernel, n):
    import bench
    r = bench.roofline_of({kernel: (200.0, 10.0, 1.5e14, 9.0e10)}, 400.0, 0, (512, 513, 64))
    peak = 152 * 30 * 2.07e9 / bench.fixed_point_madds(n) * 5 * math.log2(n) / 1e12
    assert r["fixed_point_peak"] == pytest.approx(peak)
    assert r["fixed_point_frac"] == pytest.approx(r["achieved"] / peak)


def test_other_kernels_have_no_fixed_point_figures():
    import bench
    assert "fixed_point_peak" not in bench.roofline_of({"eval": (200.0, 10.0, 1.5e14, 9.0e10)}, 400.0, 0, (512, 513, 512))
