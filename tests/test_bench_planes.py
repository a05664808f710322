"""The benchmark's count of the operations of the bit-plane form, and the fraction
of the integer peak that follows from it (no GPU)."""

import math

import pytest

import bench
from paper_2510_21105_gb300 import workloads as wl


@pytest.mark.parametrize("maxdeg", [0, 1, 4, 7, 26, 127])
def test_uncertain_levels_follow_the_thresholds(maxdeg):
    """Largest e + 1 over the m with a threshold of at least 2^24."""
    for beta in (0.0, 0.01, 0.1, 0.3, 0.9, 1.5, 2.7, 2.8, 4.0):
        m = [m for m in range(1, maxdeg + 1) if int(2.0 ** 32 * math.exp(-2 * beta * m)) >= 1 << 24]
        assert bench.msc_uncertain_levels(beta, maxdeg) == ((max(m) + 1) // 2 if m else 0)


def test_plane_operations_of_a_step():
    # 5 planes, no bonds, no threshold with a top byte: Philox 73, start and end
    # 10, upper planes 1, acceptance and tie 2, energy 15 + 12, fold 35
    assert bench.msc_plane_ops_per_attempt(0.0, 31, [3.0]) == pytest.approx((73 + 10 + 1 + 2 + 27 + 35) / 32)
    # one level: transpose, comparison, selection instead of the fold
    assert bench.msc_plane_ops_per_attempt(0.0, 31, [2.0]) == pytest.approx((73 + 10 + 1 + 2 + 27 + 64 + 9) / 32)
    # 3 planes: 13 operations per 8 bonds, 10 accumulator planes
    assert bench.msc_plane_ops_per_attempt(4.0, 4, [3.0]) == pytest.approx((73 + 6 + 6.5 + 2 + 23 + 35) / 32)


def test_roofline_reports_the_executed_form():
    stats = {"sweep_ms": 1500.0, "sweep_launches": 1000}
    probe = {"int_ops_per_s": 30e12, "philox_words_per_s": 1.6e12, "smem_bytes_per_s": 38e12, "sms": 152}
    betas = wl.linear_betas(0.1, 4.0, 50)
    attempts = 7000 * 16384 * 10
    args = (stats, attempts, probe, 2000.0, ("k_sweep_msc+pair", 256), 11.8454, 0.06)
    r = bench.sweep_roofline(*args, betas=betas)
    planes = bench.msc_plane_ops_per_attempt(11.8454, 31, betas)
    assert r["ops_per_attempt_planes"] == pytest.approx(planes)
    assert r["frac_planes"] == pytest.approx(attempts / 1.5e-3 * planes / 30e12)
    assert planes < bench.msc_ops_per_attempt(11.8454)   # "frac" counts work the kernel no longer has
    assert bench.sweep_roofline(*args)["frac_planes"] is None
    assert bench.sweep_roofline(stats, attempts, probe, 2000.0, ("k_sweep_packed", 128), 11.8, 0.06,
                                betas=betas)["frac_planes"] is None
