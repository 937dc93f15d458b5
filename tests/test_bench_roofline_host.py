"""bench.py's roofline figures for runs of steps (CPU only): the bytes of the form a run takes, the
traffic records of that form, and no fraction of the measured bandwidth above one."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

L2 = 129 << 20
PEAK = 6759.0
# Milliseconds per step of runs of 100 steps at 8192^2, as measured.
MEASURED_MS = {"f32": 0.3737, "bf16_dev": 0.4420}


@pytest.mark.parametrize("name,nx,ny,moment", [
    ("f32", 8192, 8192, True), ("f32", 512, 512, False), ("f32", 1344, 1344, False), ("f32", 1376, 1376, True),
    ("f32", 1001, 517, True), ("f32", 512, 500, True), ("f32", 7, 9, False), ("bf16_dev", 64, 64, True),
    ("f16_dev", 66, 64, False)])
def test_form_of_a_run(name, nx, ny, moment):
    assert bench.moment_form(name, nx, ny, L2) == moment


def test_bytes_of_a_run():
    assert bench.run_bytes("f32", False, 100) == 72 and bench.run_bytes("bf16_dev", False, 100) == 48
    # gather 36 + 16, 99 steps of 32, the last one 16 + 36
    assert bench.run_bytes("f32", True, 100) == (52 + 99 * 32 + 52) / 100
    assert bench.run_bytes("f16_dev", True, 100) == (36 + 99 * 24 + 36) / 100


@pytest.mark.parametrize("name", sorted(MEASURED_MS))
def test_roofline_of_the_large_field(name):
    r = bench.step_roofline(name, 8192, MEASURED_MS[name] * 1e-3, L2, PEAK, "measured")
    assert 0.3 < r["frac"] <= 1.0
    assert 0.9 * r["algorithmic_bytes_per_launch"] <= r["traffic"] <= 1.05 * r["algorithmic_bytes_per_launch"]


@pytest.mark.parametrize("name", sorted(bench.MOMENT_BYTES))
def test_moment_traffic_record_matches_current_kernel(name):
    b = bench.profiled_traffic(name, moment=True)
    assert b is not None, f"profiles/step_kernel_{name}_moment_traffic.txt is not of the current step-kernel source"
    assert 0.9 * bench.MOMENT_BYTES[name] <= b <= 1.05 * bench.MOMENT_BYTES[name]
