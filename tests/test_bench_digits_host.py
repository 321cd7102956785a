"""The roofline of products that run as exact BF16 digit products: the BF16 peak over their number."""

import pytest

import bench


@pytest.mark.parametrize("prec,phase,held,nd", [("fp64", "gemm_xv_link", True, 36), ("fp64", "gemm_xtr", True, 36),
                                                ("fp64", "cert_xtzeta", True, 36), ("bf16", "cert_xtzeta", False, 21),
                                                ("tf32x3", "cert_xtzeta", True, 21)])
def test_peak_of_digit_products(prec, phase, held, nd):
    stats = {phase: dict(ms=10.0, launches=10, work=1e11)}          # 1e10 flops per 1 ms launch: 10 TFLOP/s
    pk = {"hbm_gbs": 6792.7, "bf16_tflops_sustained": 1764.9, "source": "measured"}
    r = bench.roofline(stats, prec, pk, digits=bench.digit_products(prec, held))
    assert r["bound"] == "tensor" and r["achieved"] == pytest.approx(10.0)
    assert r["peak"] == pytest.approx(1764.9 / nd) and r["frac"] == pytest.approx(10.0 * nd / 1764.9)


def test_small_fp64_batches_stay_on_the_fp64_pipe():
    stats = {"gemm_xtr": dict(ms=10.0, launches=10, work=1e9)}
    r = bench.roofline(stats, "fp64", {"hbm_gbs": 1.0, "source": "x"}, digits=bench.digit_products("fp64", False))
    assert r["bound"] == "alu" and r["peak"] == bench.FP64_NOMINAL_TFLOPS
