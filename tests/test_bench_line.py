"""The bench line: one JSON object short enough to be recorded whole, with the
keys of the contract, whatever the workloads beside the default one report; the
details go to standard error."""
import json

import bench


def _full(workloads):
    kernel = {f"AP.symbolic.kernel_{i}": 0.123456789012345 for i in range(20)}
    roof = {"bound": "alu", "pipe": "fp64", "achieved": 0.4991790757608982, "peak": 1.25856, "unit": "TFLOP/s",
            "frac": 0.39662715783188585, "peak_source": "x" * 130,
            "hbm": {"achieved": 1121.21015405755, "peak": 6770.5, "unit": "GB/s", "frac": 0.16560226778783693, "peak_source": "measured"},
            "traffic": 1420121856, "kernel": "AP.numeric.narrow", "bytes_per_launch": 1144796832,
            "flop_per_launch": 509680208, "ms_per_launch": 1.0210368037223816}
    return {"metric": bench.METRIC, "value": 295.56093793552014, "unit": "GFLOP/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 2.4004352569580076, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic (seeded generators)",
            "config": {"workload": bench.workload_name(128), "grid": 128, "mults": 354737448, "nnz_AP": 25934336,
                       "nnz_RAP": 2048383, "l2": "inputs larger than L2 (A alone 686 MB), no flush",
                       "parallelism": "replicas x1"},
            "pct_hbm_byte_roofline": 9.924696922854103, "pct_fp64_roofline": 23.484056217861696,
            "step_algorithmic_bytes": 1612976324, "roofline": roof, "kernels_ms_per_step": kernel,
            "kernels_ms_note": "n" * 120, "gpu_launches": 180,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 6},
            "e2e": {"value": 113.18317618860945, "unit": "GFLOP/s", "h2d_bytes_per_step": 931781200,
                    "d2h_bytes_per_step": 25216660, "ms_per_step": 6.268377685546875,
                    "entry_point": "spgemm_host (A, P host -> AP device; R host * AP -> RAP host)"},
            "cpu_baseline": {"value": 8.654696356894453, "unit": "GFLOP/s", "cores": 16, "kind": "oracle",
                             "sample": "full workload (A*P then R*(AP)), median of 3 runs"},
            "secondary": workloads}


def _workload(bad=False):
    return {"metric_value": 119.70705943680622, "unit": "GFLOP/s", "ms_per_step": 1172.7020263671875,
            "config": {"workload": "w" * 150}, "kernels_ms_per_step": {str(i): 1.23456789 for i in range(30)},
            "cases": {str(i): {"parity": {"pattern_exact": True, "values_in_tolerance": not (bad and i == 3),
                                          "max_err_over_bound": 1e-16, "rows": [0, 10]}} for i in range(8)}}


def test_line_is_short_and_complete(capsys):
    full = _full({f"workload_{i}": _workload(i == 2) for i in range(6)} | {"broken": {"error": "RuntimeError: " + "x" * 500}})
    assert len(json.dumps(full)) > 3 * bench.LINE_MAX
    bench.emit(full)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) <= bench.LINE_MAX + 1
    line = json.loads(out)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "roofline", "gpu_launches", "clocks", "e2e", "cpu_baseline"):
        assert key in line, key
    assert line["config"] == full["config"] and line["clocks"] == full["clocks"] and line["gpu_launches"] == 180
    assert abs(line["value"] / full["value"] - 1) < 1e-5 and line["e2e"]["h2d_bytes_per_step"] == 931781200
    assert [d.get("ok") for d in line["secondary"].values()] == [True, True, False, True, True, True, None]
    assert json.loads(err) == full


def test_many_workloads_never_cost_the_line(capsys):
    bench.emit(_full({f"workload_{i}": _workload() for i in range(200)}))
    out = capsys.readouterr().out
    assert len(out) <= bench.LINE_MAX + 1 and json.loads(out)["value"] > 0
