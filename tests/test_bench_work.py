"""The JSON line of bench.py, and the operation counts of its FP64 rooflines against counts of the elimination."""
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def _lu_operations(m, n):
    """Multiply-adds (two operations each) of the trailing updates of one m x n LU."""
    return sum(2 * (m - j - 1) * (n - j - 1) for j in range(n))


@pytest.mark.parametrize("m,n", [(1600, 700), (700, 700), (2304, 1152)])
def test_lu_count(m, n):
    import bench

    assert bench.lu_flop(m, n) == pytest.approx(_lu_operations(m, n), rel=2.0 / n)


@pytest.mark.parametrize("Ns,n_e", [(576, 576), (400, 200)])
def test_spin_coupled_recompute_is_counted_once_per_walker(Ns, n_e):
    import bench

    got = bench.soc_recompute_flop(Ns, n_e)
    assert got["elim"] == pytest.approx(_lu_operations(4 * Ns, 2 * n_e), rel=2.0 / n_e)
    assert got["lu_o"] == pytest.approx(_lu_operations(2 * n_e, 2 * n_e), rel=2.0 / n_e)
    assert got["solve"] == 2 * (2 * n_e) ** 2 * (2 * Ns)  # a multiply-add per entry of L and U and column


def _full_line():
    """A line of the real one's shape and size: the headline's keys and some 30 KB of per-leg results."""
    import bench

    roof = {"kernel": "k" * 110, "bound": "tensor", "achieved": 212.31836211834784, "peak": 1922.5, "unit": "TFLOP/s",
            "frac": 0.11043867990551252, "traffic": None, "launches": 192, "ms_per_launch": 0.9495174981032809,
            "ms_per_step": 91.15367981791496, "work_per_launch": 201600000000.0, "fp64_equivalent_tflops": 4.718,
            "fp64_equivalent_vs_fp64_peak": 4.2978, "peak_source": "s" * 130}
    return {"metric": bench.METRIC, "value": 573811.9719297137, "unit": bench.UNIT, "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": 446.13917541503906, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic", "config": bench.arm_config(64),
            "update_only": {"value": 1.0}, "speedup_update_only_vs_local": {"delayed": 3.25431, "blockfb": 2.72313},
            "G_err_fp32_vs_fp64_recompute": {"max": 1.0e-2, "median": 4.2e-4, "slices_between_recomputes": 5,
                                             "tolerance_median": 1e-3, "within_tolerance": True, "note": "n" * 150,
                                             "by_point": [{"slice": 5, "dir": 1, "drift": 4.2e-4}] * 96},
            "roofline": roof, "roofline_kernels": [roof] * 8,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 62}, "gpu_launches": 36480,
            "e2e": {"value": 471991.123456789, "unit": bench.UNIT, "h2d_bytes_per_step": 18048000,
                    "d2h_bytes_per_step": 128016, "note": "n" * 90},
            "soc": {"modes": [roof] * 12}, "precision_report": {"x": list(range(1000))},
            "cpu_baseline": {"value": 2596.389029112185, "unit": bench.UNIT, "cores": 16, "kind": "oracle",
                             "sample": "s" * 150}}


def test_stdout_line_fits_the_end_of_a_log():
    """The line of stdout alone, whole within the last 3000 characters, with the workload's result in it."""
    import bench

    full = _full_line()
    text = json.dumps(bench.headline(full))
    assert len(text) < 2800 < len(json.dumps(full)) and "\n" not in text
    got = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "gpu_launches", "e2e", "clocks", "roofline", "cpu_baseline"):
        assert got[key] == full[key], key
    assert got["G_err_fp32_vs_fp64_recompute"]["median"] == 4.2e-4
