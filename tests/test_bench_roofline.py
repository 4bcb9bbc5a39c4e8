"""The FP64 roofline of the bench counts the time of every kernel that evaluates walkers."""
import pytest

import bench


def test_fp64_roofline_includes_the_step_kernels(monkeypatch):
    """Small problems evaluate their walkers inside the step kernel (class 3): 1.4e6 evaluations
    at d = 64, K = 4 in 32 ms there and 5 ms of the likelihood kernels (classes 4, 5)."""
    monkeypatch.setattr(bench, "fp64_peak", lambda sb: {"tflops": 1.0})
    ms = [0.0, 0.0, 0.0, 64.0, 9.6, 0.4, 0.1, 0.0]  # two steps
    r = bench.fp64_roofline(None, ms, [6] * 8, 2, 1.4e6, 64, 4)
    flop = 1.4e6 * 2 * 4 * 64 * 65
    assert r["achieved"] == pytest.approx(flop / 37e-3 / 1e9)
    assert r["frac"] == pytest.approx(r["achieved"] / 1e3)


def test_factorizations_of_a_group_of_modes_share_a_launch():
    """Two modes at d = 1024 factored in one launch of 1.5 ms."""
    r = bench.factorization_rate(1024, 2, 1, 1.5, 1.0)
    assert r["factorizations"] == 2 and r["launches"] == 1 and r["ms_per_launch"] == 1.5
    assert r["frac"] == r["fp64_TFLOPs"] == pytest.approx(2 * 1024 ** 3 / 3 / 1.5e-3 / 1e12)
    assert bench.factorization_rate(1024, 2, 0, 0.0, 1.0) == {"factorizations": 0, "launches": 0}
