"""The bench's printed line: short enough to be read back from the end of a
program's output, with every key a reader needs, and the whole record beside
it."""
import json
import os

import bench


def record():
    """The saved record of a whole run."""
    path = os.path.join(os.path.dirname(bench.__file__), "profiles",
                        "bench_short_sweep_30M.json")
    with open(path) as f:
        return json.loads(f.read().strip().splitlines()[-1])


def test_line_is_short_and_whole_record_is_kept(tmp_path, capsys):
    line = record()
    path = str(tmp_path / "sub" / "details.json")
    bench.print_line(line, path)
    out = capsys.readouterr().out
    assert out.count("\n") == 1 and len(out) < 8000
    short = json.loads(out)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup",
                "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
                "dtype", "data", "config", "clocks", "e2e", "gpu_launches"):
        assert short[key] == line[key], key
    with open(path) as f:
        assert json.load(f) == line
    assert os.path.normpath(os.path.join(os.path.dirname(bench.__file__),
                                         short["details"])) == path
    assert len(json.dumps(line)) > 16000  # (which is what was printed)


def test_line_without_a_place_for_the_record(tmp_path, capsys):
    blocked = tmp_path / "file"
    blocked.write_text("")
    bench.print_line({"value": 1.0}, str(blocked / "details.json"))
    got = capsys.readouterr()
    assert json.loads(got.out) == {"value": 1.0}
    assert "not written" in got.err
