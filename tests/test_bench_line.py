"""The benchmark's result line stays short whatever the sweep was, and is the last thing on stdout."""
import importlib.util
import json
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sweep_goes_to_stderr(capsys):
    spec = importlib.util.spec_from_file_location("bench_mod", os.path.join(ROOT, "bench.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    sweep = [{"variant": "greedy_es", "es_vl": 20, "beam": k, "ap": 0.123456789, "ms": 1.0 / 3, "qps": 1e6 / 3}
             for k in range(400)]
    b.emit({"metric": "range QPS at AP>=0.95", "value": 1.0}, sweep)
    out, err = capsys.readouterr()
    assert json.loads(out) == {"metric": "range QPS at AP>=0.95", "value": 1.0}
    assert err.count("sweep") == 400 and '"ap": 0.12346' in err


def test_the_line_holds_no_sweep():
    src = open(os.path.join(ROOT, "bench.py")).read()
    assert "emit(line, sweep)" in src and '"sweep":' not in src
