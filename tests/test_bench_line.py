"""The roofline of a bench line (CPU only): the traffic is that of the kernels that ran, and no fraction is given
against a pipe that the work does not run on."""
from types import SimpleNamespace

import bench

W = SimpleNamespace(n_traj=1024, nx=1024, nR=512)
PEAKS = {"hbm_gbs": 6700.0, "bf16_tflops_sustained": 1700.0}


def test_traffic_of_the_present_factorisation():
    r = bench.line_roofline({"cholesky": (94.0, 100)}, W, 1, "tf32x3", PEAKS)
    assert r["traffic"] == 63.9e6 and "launches_mixed_and_fp64_N1024" in r["traffic_source"]
    # other arithmetic, one matrix per call, or another family: not measured
    assert bench.line_roofline({"cholesky": (94.0, 100)}, W, 1, "tf32x3", PEAKS, "fp64")["traffic"] is None
    assert bench.line_roofline({"cholesky": (94.0, 100)}, W, 1, "tf32x3", PEAKS, "df64", 1)["traffic"] is None
    assert bench.line_roofline({"assemble": (94.0, 100)}, W, 1, "tf32x3", PEAKS)["traffic"] is None


def test_no_fraction_of_the_fp64_pipe_for_digit_products():
    for fam in ("assemble", "cholesky"):
        r = bench.line_roofline({fam: (300.0, 100)}, W, 21, "fp64", PEAKS)
        assert r["achieved"] > 0 and r["frac"] is None
    assert bench.line_roofline({"cholesky": (94.0, 100)}, W, 21, "bf16x3", PEAKS, "fp64")["frac"] is None
    assert bench.line_roofline({"chol_solve": (94.0, 100)}, W, 21, "fp64", PEAKS)["frac"] < 1
    assert bench.line_roofline({"assemble": (108.0, 100)}, W, 16, "tf32x3", PEAKS)["frac"] < 1
