"""The benchmark's printed line: one line of strict JSON, short whatever the sections hold."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_line_is_short_and_strict(tmp_path, capsys):
    sys.path.insert(0, ROOT)
    import bench
    runs = [{"scheme": "two", "kappa": 1e14, "orth_err": float("nan"), "ms": 1.5, "status": 4}] * 400
    line = {"metric": bench.METRIC, "value": 0.17, "unit": "s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 340.0, "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": bench.WORKLOAD, "n": 10 ** 6}, "gpu_launches": 7,
            "solves": {"one_stage": {"iterations": 860, "relres": float("inf")}},
            "roofline": {"bound": "hbm", "frac": 0.3, "traffic": {"rows": runs}},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "e2e": {"value": 0.17, "unit": "s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
            "cpu_baseline": {"value": 46.0}, "orth": {"runs": runs}, "stress": runs}
    path = tmp_path / "sections.json"
    bench.emit(line, str(path))
    text = capsys.readouterr().out
    assert text.count("\n") == 1 and len(text) < 3000

    def no_constant(name):
        raise AssertionError(name)

    got = json.loads(text, parse_constant=no_constant)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert got[k] == line[k]
    assert got["solves"]["one_stage"]["relres"] is None
    full = json.loads(path.read_text(), parse_constant=no_constant)
    assert len(full["orth"]["runs"]) == 400 and full["orth"]["runs"][0]["orth_err"] is None
    bench.emit(line, "")
    assert "sections" not in json.loads(capsys.readouterr().out)
