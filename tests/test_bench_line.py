"""The bench's printed line: one JSON object that is short enough to be read
from the end of an output, with every field of the contract; the complete
record goes to a file."""
import json

import bench

CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks")


def record(subs):
    roof = {"bound": "tensor", "achieved": 380.48508255175733, "peak": 1935.3, "unit": "TFLOP/s",
            "frac": 0.196602636568882, "kernel": "mqo::k_step_t", "step_kernel_ms": 0.10532607898116111,
            "peak_derivation": "x" * 200, "hbm": {"achieved": 1.0}, "plan": {"dense": True}}
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 30}
    line = {"metric": "edge-updates/s of fused mQO steps; HBM GB/s vs peak; best MIS/cut vs oracle",
            "value": 9925462789321.123, "unit": "edge-updates/s", "n_gpus": 1, "steps": 200, "warmup": 20,
            "ms_per_step": 0.13640000000000002, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32 (x bf16 / V bf16 storage, int64 evaluation)", "data": "synthetic",
            "config": {k: "y" * 100 for k in ("workload", "value_counts", "l2")},
            "e2e": {"value": 6953777782518.533, "unit": "edge-updates/s", "h2d_bytes_per_step": 878256,
                    "d2h_bytes_per_step": 131072, "note": "z" * 150},
            "gpu_launches": 1000, "clocks": clocks, "roofline": roof, "best_mean": 41.6, "best_max": 46,
            "kernel_ms_per_step": {p: 0.011361919920891523 for p in ("ctrl", "apply", "step", "disc_a", "tick_end")},
            "cpu_baseline": {"value": 12219684068.634956, "cores": 16, "kind": "oracle", "sample": "s" * 250}}
    line["steady_state"] = {"value_median": 9637528503686.523, "ms_per_step_median": 0.142, "clocks": clocks}
    line["configs"] = {f"workload_{k}_with_a_long_name": dict(line, roofline=dict(roof)) for k in range(subs)}
    line["paper_er"] = {"best_per_graph": [1.0] * 500}
    return line


def test_line_is_short_and_complete(capsys, tmp_path):
    for subs in (0, 7, 60):
        line = record(subs)
        path = tmp_path / "detail.json"
        bench.emit(line, str(path))
        out = capsys.readouterr().out
        assert out.count("\n") == 1 and len(out) <= bench.LINE_LIMIT
        got = json.loads(out)
        for k in CONTRACT:
            if k == "e2e":
                assert {a: b for a, b in line[k].items() if a != "note"} == got[k]
            else:
                assert got[k] == line[k], k
        assert json.loads(path.read_text()) == line
        if subs == 7:  # value and time of every sub-record
            assert len(got["configs"]) == 7
            assert all(v == {"value": 9.92546e12, "ms_per_step": 0.1364} for v in got["configs"].values())


def test_line_without_a_place_for_the_record(capsys, tmp_path):
    bench.emit(record(2), str(tmp_path / "missing" / "detail.json"))
    assert json.loads(capsys.readouterr().out)["value"] == record(2)["value"]
