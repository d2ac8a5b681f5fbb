"""The benchmark's roofline of one-kernel passes (window plan and sums in one launch), whose launches are
timed in the plan's class: their bound is the work they do, not a plan's traffic."""
from types import SimpleNamespace

import pytest

import bench


def _roof(plan_launches, window_launches, work, n=256, iters=100):
    ktimes = {"band_plan_kernel": (4.0, plan_launches), "band_pass_kernel": (1.0 * (window_launches > 0), window_launches),
              "tc_pass_kernel": (0.0, 0), "axis_pass_kernel": (0.0, 0)}
    return bench._roofline(n, SimpleNamespace(steps=1, iters=iters, precision="fp32"), ktimes, work, 5.0)


def test_exact_passes_are_bound_by_exponentials():
    terms = 2.0e9
    r = _roof(400, 0, (0.0, terms, 0.0, 0.0))
    assert r["bound"] == "alu" and r["unit"] == "Tex2/s"
    assert r["achieved"] == pytest.approx(terms / 4e-3 / 1e12)


def test_product_passes_are_bound_by_the_tensor_cores():
    r = _roof(400, 0, (2.0e9, 1.0e6, 0.0, 0.0))
    assert r["bound"] == "tensor" and r["achieved"] == pytest.approx(6.0 * 2.0e9 / 4e-3 / 1e12)


def test_passes_with_few_terms_are_bound_by_both_images():
    r = _roof(400, 0, (1.0e3, 1.0e3, 0.0, 0.0))
    assert r["bound"] == "hbm" and r["achieved"] == pytest.approx(400 * 2 * 256 * 256 * 4 / 4e-3 / 1e9)


def test_plans_beside_window_kernels_are_bound_by_their_traffic():
    r = _roof(400, 400, (2.0e9, 0.0, 0.0, 0.0))
    assert r["bound"] == "hbm" and r["achieved"] == pytest.approx(400 * (256 * 256 * 4 + 256 * 16 * 12) / 4e-3 / 1e9)
