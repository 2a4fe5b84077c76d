"""The benchmark line's roofline counts the operations that the kernels execute and
names the kernels that ran."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_executed_operations_and_kernel_names():
    stats = {"inter2_items": 4, "pair2_items": 0, "cells": 10 ** 12, "inter_cells": 9 * 10 ** 11}
    t = {"stats": stats, "kernel_ms": [100.0], "pair_ms": [20.0], "recompute_ms": [0.01]}
    r = bench.executed_roofline(bench.roofline(t, 20.0, "test", 2070.0, lambda k: None))
    # packed_cell, two queries per word: 3.5 ALU operations for two cells
    assert r["alu_ops_per_cell"] == 1.75 and abs(r["achieved"] - 1.75 * 9e11 / 0.1 / 1e12) < 1e-3
    assert abs(r["frac"] - r["achieved"] / 20.0) < 1e-4
    assert abs(r["peak_gcups"] - 20.0e3 / 1.75) < 0.1
    assert abs(r["yardstick"]["frac"] / r["frac"] - 2.25 / 1.75) < 1e-3
    # two subjects per word: 4.5, by the kernel that runs
    lanes = [k for k in r["kernels"] if k.startswith("lane_kernel (long subjects")]
    assert len(lanes) == 1 and not any("pair_kernel" in k for k in r["kernels"])
    assert r["kernels"][lanes[0]]["alu_ops_per_cell"] == 2.25
    assert abs(r["kernels"][lanes[0]]["achieved"] - 2.25 * 1e11 / 0.02 / 1e12) < 1e-3
