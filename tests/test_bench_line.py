"""The benchmark's record as one short line on stdout (no GPU): readers keep
the last kilobytes of the output, so the line has to fit them whole; the full
record goes to stderr."""
import json

import bench


def full_record():
    note = "counted per walker over the live basis rows of the final positions; " * 4
    roof = {"kernel": "k_sweep64", "bound": "alu", "achieved": 0.123456789012, "peak": 1.25, "unit": "TFLOP/s",
            "frac": 0.098765432101, "traffic": None, "flops_counted": note, "peak_source": note}
    rate = {"value": 6278319.8823599545, "unit": "electron-moves/s", "ms_per_step": 9.8765432101,
            "force_evals_per_s": 104231.15290448, "roofline": roof, "roofline_force": roof,
            "error_vs_oracle": {f"quantity_{k}": 1.0 / (k + 3) for k in range(20)}, "recompute": {"what": note},
            "config": {"what": note}, "cpu_baseline": {"sample": note}}
    cfg = {f"key_{k}": "a value of some length" for k in range(16)}
    return {"metric": bench.METRIC, "n_gpus": 1, "steps": 20, "warmup": 5, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", **rate, "config": cfg, "gpu_launches": 100,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 3},
            "e2e": {"value": 6.1e6, "unit": "electron-moves/s", "h2d_bytes_per_step": 147456.0,
                    "d2h_bytes_per_step": 147523.2, "what": note[:140]},
            "cpu_baseline": {"value": 5000.123456, "unit": "electron-moves/s", "cores": 16, "kind": "oracle",
                             "sample": note},
            "kernel_ms_per_step": {k: 1.23456789012 for k in ("sweep", "eloc", "force", "branch", "reduce", "all")},
            "mixed": rate, "workloads": {n: rate for n in ("water32_mixed", "batch64_uneven", "water32_pp", "water6_pp")},
            "space_warp": rate}


def test_headline_is_short_and_keeps_the_rates(capsys):
    rec = full_record()
    assert len(json.dumps(rec)) > 9000
    bench.emit(rec)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) <= bench.HEADLINE_BYTES + 1
    line = json.loads(out)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "force_evals_per_s"):
        assert line[k] == rec[k], k
    assert line["roofline"]["kernel"] == "k_sweep64" and line["cpu_baseline"]["kind"] == "oracle"
    assert set(line["workloads"]) == set(rec["workloads"])
    assert json.loads(err) == rec


def test_headline_never_drops_the_contract():
    rec = full_record()
    rec["workloads"] = {f"workload_{k}": rec["mixed"] for k in range(200)}
    line = bench.headline(rec)
    assert "workloads" not in line and line["value"] == rec["value"] and line["e2e"] == rec["e2e"]
