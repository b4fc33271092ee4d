"""bench.py's FP64 roofline: the instruction count fits the kernel it is applied to."""
import pytest

bench = pytest.importorskip("bench")


def test_fp64_fraction_is_of_the_kernel_that_runs():
    # 2048 x 1024 in 286.2 us (profiles/k_collide_stream_fp64_alu.md): ncu saw the FP64 pipe
    # active for 85 % of the cycles
    r = bench.fp64_roofline(2048 * 1024 / 286.2e-6 / 1e9, 2070.0)
    assert abs(r["frac"] - 0.85) < 0.02


def test_a_fraction_above_one_is_not_reported():
    r = bench.fp64_roofline(1.01 * 304 * 2.070 / bench.FP64_INSTR_PER_UPDATE, 2070.0)
    assert r["frac"] is None and "error" in r
    assert bench.fp64_roofline(0.99 * 304 * 2.070 / bench.FP64_INSTR_PER_UPDATE, 2070.0)["frac"] < 1.0
