"""The bench's roofline of the forms on the CUDA cores: a rate and a fraction of the peak only
where every pair is evaluated, so that work left out is never counted as done."""
import pytest


@pytest.mark.parametrize("r,n,prec,full", [(1000, 2000, "f32", False), (128, 513, "f32", False), (127, 65536, "f32", True),
                                           (128, 512, "f32", True), (511, 300, "f32", True), (512, 300, "f32", False),
                                           (1000, 65536, "f32s", False), (100, 16384, "f32s", False),
                                           (100, 2048, "f32s", True), (63, 65536, "f32s", True),
                                           (2, 1024, "f64", False), (65, 1024, "f64", False)])
def test_no_fraction_where_terms_are_left_out(r, n, prec, full):
    import bench
    roof = bench._alu_roofline(r, n, prec, 0.01)   # 10 us
    if full:
        assert roof["achieved"] == pytest.approx(3.0 * n * n * r / 1e-5 / 1e12, rel=1e-3, abs=1e-3)
        assert roof["peak"] > 0 and roof["algorithmic_flops_per_launch"] == 3.0 * n * n * r
        assert bench._takes_every_pair(r, n, prec)
    else:
        assert roof["achieved"] is None and roof["peak"] is None and "algorithmic_flops_per_launch" not in roof
