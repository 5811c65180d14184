"""The benchmark's printed line: every key its readers need, in a few
kilobytes, whatever the side measurements hold; the whole record in a file."""
import json

import bench


def _record():
    side = {"k%d" % i: {"greeks_per_s": 1.0 / 3, "text": "x" * 400} for i in range(60)}
    return {
        "metric": "Greeks/s", "value": 668.7256865519771, "unit": "Greeks/s", "n_gpus": 1,
        "steps": 20, "warmup": 5, "ms_per_step": 37.38453674316406, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "w" * 60, "n_paths": 131072, "n_steps": 252,
                   "strikes": [80.0] * 5, "greeks": ["delta"] * 5, "l2": "x" * 60},
        "path_steps_per_s": {"generated": 1e9 / 3, "lsmc": 1e10 / 3},
        "max_rel_err_vs_oracle": 3.7e-11 / 3, "accuracy_ok": True,
        "roofline": {"kernel": "backward_kernel", "bound": "issue", "achieved": 22.0 / 3,
                     "peak": 39.3, "unit": "Tinst/s", "frac": 0.57, "kernel_ms": {"a": 1.0 / 3},
                     "algorithmic_tflops": 1.9, "traffic": 5.4e9, "stepper": side},
        "cpu_baseline": {"value": 1.0 / 3, "sample": "y" * 300},
        "e2e": {"value": 667.4, "unit": "Greeks/s", "h2d_bytes_per_step": 18688,
                "d2h_bytes_per_step": 3496}, "gpu_launches": 80,
        "clocks": {"sm_mhz": 2070, "sm_max_mhz": 2070, "reasons": []}, "device_bytes": 10**10,
        "precision_split": side, "serving_curve": side,
        "greeks_per_s_within_1e-4": {"forms": side, "best": "book.df", "best_greeks_per_s": 2193.9,
                                     "outside_1e-4": side},
    }


def test_the_line_is_short_and_whole():
    rec = _record()
    assert len(json.dumps(rec)) > 60000
    text = json.dumps(bench.printed_line(rec))
    assert len(text) < 4000 and "\n" not in text
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
              "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "e2e",
              "gpu_launches", "clocks"):
        assert line[k] == rec[k], k
    assert line["roofline"]["frac"] == 0.57 and "stepper" not in line["roofline"]


def test_the_details_hold_the_whole_record(tmp_path, monkeypatch, capsys):
    rec = _record()
    monkeypatch.setattr(bench, "DETAILS", str(tmp_path / "d.json"))
    bench.write_details(rec)
    assert json.load(open(tmp_path / "d.json")) == rec
    monkeypatch.setattr(bench, "DETAILS", str(tmp_path / "no" / "d.json"))
    bench.write_details(rec)  # no such folder: said, not raised
    assert capsys.readouterr().out == ""
