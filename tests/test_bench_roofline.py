"""bench.py's float64 roofline names the unit that the products ran on."""
import pytest

import bench

PK = {"bf16_tflops_sustained": 1700.0}


def test_digit_products_against_the_tensor_peak():
    acc = {"tensor_flops": 3.4e12, "prod_s": 0.004, "useful": 8e10, "mults": 20}
    r = bench.fp64_roofline(acc, PK, "measured", 2000.0)
    assert r["bound"] == "tensor" and r["frac"] == pytest.approx(0.5) and "f64_digit_product" in r["kernel"]


def test_the_fma_kernel_against_the_float64_pipe():
    # n < 160, n > 32768, an operand or a density that digits cannot hold
    acc = {"tensor_flops": 0.0, "prod_s": 0.1, "useful": 6.08e10, "mults": 20}
    r = bench.fp64_roofline(acc, PK, "measured", 2000.0)
    assert r["bound"] == "alu" and r["kernel"] == "step_f64_kernel"
    assert r["peak"] == pytest.approx(152 * 4 * 2e9 / 1e12) and r["frac"] == pytest.approx(0.5)
