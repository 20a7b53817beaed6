"""The bench's result line: one JSON line on standard output that carries the keys of the contract and
stays short enough to be read from the end of a log (the record with every table and sub-record is
tens of kilobytes and goes to standard error or the file named by --detail, from which --plan-from
takes its plan)."""
import importlib.util
import json
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

KEYS = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
        "dtype", "data", "config", "e2e", "gpu_launches", "clocks")


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_module", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def _record(value):
    classes = {"rbgs_split_f64@%d" % n: {"launches": 123, "ms": 1.0 / 3.0, "share": 1.0 / 7.0} for n in range(60)}
    return {
        "metric": "MLMC samples/s (all levels, c2_mlmc4_f64)", "value": value, "unit": "samples/s", "n_gpus": 8, "steps": 20,
        "warmup": 5, "ms_per_step": 1000.0 / 3.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64", "solver": {"precision": "f64"}, "plan": {"autotune": {"0": {"best": {"smoother": "split", "nu": 2}}}},
        "data": "synthetic (seeded Philox realisations, run_seed 1607032520)",
        "config": {"workload": "c2_mlmc4_f64", "levels": [0, 1, 2, 3], "N_per_gpu": [4096, 1024, 256, 64],
                   "fine_n": [17, 33, 65, 129], "sigma2": 1.0, "ell": 0.3, "M": 256, "rtol": 1e-10, "cycle": "V(2,2)",
                   "parallelism": "replicas x8 (samples sharded by rank, no data-path collective)",
                   "level_streams": [["%d[%d:%d]" % (l, 0, 4096) for l in range(9)]] * 4,
                   "level_ms_alone": {str(l): 1.0 / 3.0 for l in range(4)}, "level_launches_alone": {str(l): 700 for l in range(4)},
                   "l2": "every level's batch working set exceeds the 129 MB L2 (no flush needed)"},
        "per_level": {str(l): 1.0 / 3.0 for l in range(4)}, "roofline": {"kernel": "rbgs_split_f64@129", "bound": "alu",
        "achieved": 1.0 / 3.0, "peak": 1.25856, "unit": "TFLOP/s", "frac": 0.8324450504701539, "traffic": None},
        "gpu_launches": 26040, "e2e": {"value": 19737.26587597166, "unit": "samples/s", "h2d_bytes_per_step": 43520,
        "d2h_bytes_per_step": 130560, "api": "mlmc_level_estimate (host ids in, Y/Qf/Qc to pinned host memory)"},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 7},
        "cpu_baseline": {"value": 39.823121996147805, "unit": "samples/s", "cores": 16, "kind": "oracle", "sample": "x" * 300},
        "kernel_classes": classes, "c3": {"value": 4280.0 / 3.0, "unit": "samples/s", "kernel_classes": classes},
        "c4": {"value": 85.6, "unit": "samples/s", "serving_sweep": [classes]}, "c5": {"value": 1.1 / 3.0, "unit": "s"},
        "c6": {"value": 83645.0 / 7.0, "unit": "samples/s", "plan": classes}}


def test_line_is_short_and_complete(bench, capsys, tmp_path):
    full = _record(19402.123456789)
    detail = tmp_path / "detail.json"
    bench.report(full, str(detail))
    out, err = capsys.readouterr()
    lines = [ln for ln in out.splitlines() if ln.strip()]
    assert len(lines) == 1 and len(lines[0]) < 1500
    line = json.loads(lines[0])
    for key in KEYS:
        assert key in line, key
        if key not in ("config", "e2e", "clocks"):
            assert line[key] == full[key]
    for key in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][key] == full["e2e"][key]
    for key in ("sm_mhz", "sm_max_mhz", "reasons"):
        assert line["clocks"][key] == full["clocks"][key]
    for key in ("workload", "levels", "N_per_gpu", "fine_n", "sigma2", "ell", "M", "rtol", "parallelism", "l2"):
        assert line["config"][key] == full["config"][key]
    assert json.loads(detail.read_text()) == full and json.loads(err) == full


def test_sub_workloads_keep_their_lines(bench, capsys):
    bench.report({"metric": "m", "value": 1.0, "unit": "s", "arms": {"fast": "x" * 4000}, "plan": {}}, None)
    line = json.loads(capsys.readouterr().out)
    assert line["metric"] == "m" and line["value"] == 1.0 and "arms" not in line
