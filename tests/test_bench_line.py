"""The default run's standard output is the bench line alone; its studies go to standard error."""
import importlib.util
import json
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_line_alone_on_stdout(capsys):
    spec = importlib.util.spec_from_file_location("bench_module", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod.emit({"metric": mod.METRIC, "value": 1.0}, {"ess": {"chains": [0.5] * 10000}})
    out, err = capsys.readouterr()
    assert json.loads(out) == {"metric": mod.METRIC, "value": 1.0} and out.count("\n") == 1
    assert json.loads(err)["studies"]["ess"]["chains"][0] == 0.5
