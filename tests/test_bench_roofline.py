"""Roofline object of the bench from the work that the timed passes launched (no GPU)."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

PK = {"hbm_gbs": 7000.0, "bf16_tflops": 2000.0, "bf16_tflops_sustained": 1800.0}
ALGO = {"flops": 1e9, "bytes": 4e9, "factor_entries": 1}


def roofline(work, ms=20.0):
    tm = {"f_apply_ms_total": ms, "f_apply_launches": work["passes"]}
    return bench.pass_roofline(tm, work, ALGO, PK, "measured", 1.0)


def test_digit_products_alone_are_tensor_work():
    r = roofline({"passes": 100, "banded_passes": 0, "digit_flops": 14e12, "banded_flops": 0.0})
    assert r["bound"] == "tensor"
    assert r["achieved"] == pytest.approx(700.0) and r["frac"] == pytest.approx(0.35)
    assert r["executed_flops_per_launch"] == {"bf16_digit": pytest.approx(14e10), "fp64_banded": 0.0}
    assert r["fp64_method"]["achieved"] == pytest.approx(5.0)


def test_a_pass_with_banded_boxes_is_not():
    r = roofline({"passes": 100, "banded_passes": 1, "digit_flops": 14e12, "banded_flops": 4e9})
    assert r["bound"] == "alu" and r["achieved"] == pytest.approx(0.2) and r["peak"] == 1.0
    assert r["digit_product"]["achieved"] == pytest.approx(700.0)
    assert r["executed_flops_per_launch"]["fp64_banded"] == pytest.approx(4e7)


def test_no_digit_products():
    r = roofline({"passes": 10, "banded_passes": 10, "digit_flops": 0.0, "banded_flops": 1e10})
    assert r["bound"] == "alu" and r["achieved"] == pytest.approx(0.5) and r["digit_product"] is None


def test_nothing_timed():
    r = roofline({"passes": 0, "banded_passes": 0, "digit_flops": 0.0, "banded_flops": 0.0}, ms=0.0)
    assert r["achieved"] is None and r["frac"] is None
