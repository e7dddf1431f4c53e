"""bench.py's line on stdout is short enough to be read whole and keeps the
keys that identify the measurement; the whole record goes to stderr."""
import json

import bench


def test_line_is_short_and_complete(capsys):
    deep = {"value": 1.0, "unit": "u", "config": {"a": ["x" * 400] * 20}, "kernels": [{"k": i} for i in range(500)]}
    line = {"metric": bench.METRIC, "value": 2.5, "unit": "cell-updates/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.4, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": bench.config(128), "gpu_launches": 120,
            "e2e": {"value": 2.0, "unit": "u", "h2d_bytes_per_step": 8, "d2h_bytes_per_step": 8},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 9},
            "deep_amr": deep, "amr": deep, "serving": deep, "notes": ["y" * 9000]}
    bench.emit(line)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 8000
    got = json.loads(out)
    for k in line:
        if k not in ("deep_amr", "amr", "serving", "notes"):
            assert got[k] == line[k], k
    assert got["amr"] == {"value": 1.0, "unit": "u"}
    assert json.loads(err) == line
    bench.emit(line, to_stdout=True)
    assert json.loads(capsys.readouterr().out) == line
