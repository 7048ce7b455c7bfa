"""The memory bound that a bench line names: HBM for a walk in the workspace, shared memory
for one on chip, whose node values do not reach HBM."""
import pytest

import bench


def test_workspace_walk_is_held_against_hbm():
    # medium graph, FP32, 65,536 samples in 2.35 ms: 18,498 nodes written and read once
    r = bench.memory_roofline(1, False, 46188, 18498, 65536, 10, 2.35e-3, False, 1.0, 152)
    assert r["bound"] == "hbm" and r["traffic"] == 1.0
    assert r["algorithmic_bytes_per_launch"] == 65536 * (2 * 18498 * 4 + 88)
    assert r["achieved"] == pytest.approx(65536 * (2 * 18498 * 4 + 88) / 2.35e-3 / 1e9)
    both = bench.memory_roofline(1, True, 46188, 18498, 65536, 10, 2.35e-3, False, None, 152)
    assert both["algorithmic_bytes_per_launch"] == 65536 * (4 * 18498 * 4 + 96)


@pytest.mark.parametrize("mode,with_abs,operands", [(0, False, 16), (1, False, 8), (1, True, 12), (2, False, 8)])
def test_on_chip_walk_is_held_against_shared_memory(mode, with_abs, operands):
    r = bench.memory_roofline(mode, with_abs, 46188, 18498, 65536, 10, 1.62e-3, True, None, 152)
    assert r["bound"] == "smem" and r["traffic"] is None
    assert r["operand_bytes_per_launch"] == 46188 * 65536 * operands
    assert r["peak"] == pytest.approx(128 * 152 * bench_clock_ghz(), rel=1e-12)
    assert r["frac"] < 1.0   # medium count (1.87 ms at the same 8 bytes) was printed as 1.56 of HBM


def bench_clock_ghz():
    import json
    import os
    try:
        with open(os.path.join(os.path.dirname(bench.__file__), "MEASURED_PEAKS.json")) as f:
            return json.load(f)["sm_max_mhz"] / 1e3
    except OSError:
        return 2.07
