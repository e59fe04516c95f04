"""The operation counts of the bench's per-kernel model lie at or below the
instructions that the hardware counted (profiles/executed_ops.json): a count
above what a kernel executes would report a rate that it does not reach. 0.1 %
for the rounding of the recorded totals."""
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

ROWS = json.load(open(os.path.join(ROOT, "profiles", "executed_ops.json")))["rows"]


@pytest.mark.parametrize("row", ROWS, ids=lambda r: r["step"].replace(" ", "") + "-" + "+".join(r["kernels"]))
def test_model_at_or_below_the_counters(row):
    model = bench.KERNEL_MODEL if row["step"].startswith("2D") else bench.KERNEL_MODEL_3D
    assert all(model[k][2] == row["precision"] for k in row["kernels"])
    ops = sum(model[k][1] * c for k, c in zip(row["kernels"], row["cells"]))
    assert ops <= 1.001 * row["f64" if row["precision"] == "f64" else "f32"]


def test_every_kernel_of_the_model_has_a_counter_or_is_named():
    # kernels that the profiled steps do not launch: one-level solves, LES
    other = {"rb_start", "mx_rb_start", "cg_update_single", "mx_update_single", "g3_les"}
    counted = {k for r in ROWS for k in r["kernels"]}
    assert set(bench.KERNEL_MODEL) | set(bench.KERNEL_MODEL_3D) == counted | other
