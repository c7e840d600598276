"""The benchmark's line on the CPU: the headline's keys in a line short enough for a reader that
keeps the last 3,000 characters of the output, the other legs' records beside it."""
import importlib.util
import json
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def full_line():
    x = 0.1234567890123456
    leg = {"value": 1.0962282050562156e12, "seconds": x, "roofline_frac": x, "tuning": {str(i): x for i in range(80)}}
    names = ["single", "single_heun", "single_xorshift", "uneven", "heun", "xorshift", "snapshots_slice", "snapshots"]
    return {"metric": "particle-steps/s", "value": 1.0962282050562156e12, "unit": "particle-steps/s", "n_gpus": 1,
            "steps": 20, "warmup": 5, "ms_per_step": 191.30615234375, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic", "config": {"text": "x" * 500},
            "roofline": {"text": "x" * 480}, "cpu_baseline": {"text": "x" * 300},
            "e2e": {"value": 1.0946805467402953e12, "unit": "particle-steps/s", "h2d_bytes_per_step": 278944,
                    "d2h_bytes_per_step": 2228224},
            "gpu_launches": 20, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 5},
            "adjoint": {"forward_ms": 95.88310241699219, "backward_ms": 242.816162109375, "windowed": {"text": "x" * 3800}},
            "visualisation": {"text": "x" * 4000},
            "configs": dict({n: leg for n in names}, items=[{"work_items": i, "value": x} for i in range(60)],
                            precision={"rows": [x] * 60}),
            "wall_s_timed": x, "sm_count": 152, "device": "NVIDIA GB300"}


def test_the_line_is_short_and_keeps_the_contract(bench, capsys):
    line = full_line()
    assert len(json.dumps(line)) > 16000
    bench.print_line(line)
    out = capsys.readouterr()
    printed = out.out.splitlines()
    assert len(printed) == 1 and len(printed[0]) < 2900
    got = json.loads(printed[0])
    for k in line:
        if k not in bench.DETAIL_KEYS:
            assert got[k] == line[k], k
    assert got["legs"]["uneven"] == line["configs"]["uneven"]["value"]
    assert got["legs"]["adjoint"] == {"forward_ms": 95.88310241699219, "backward_ms": 242.816162109375}
    detail = json.loads(out.err.splitlines()[-1])["detail"]
    assert detail == {k: line[k] for k in bench.DETAIL_KEYS}


def test_detail_file_and_skipped_legs(bench, capsys, tmp_path):
    line = full_line()
    path = str(tmp_path / "detail.json")
    bench.print_line(line, path)
    assert capsys.readouterr().err == ""
    assert json.load(open(path)) == {k: line[k] for k in bench.DETAIL_KEYS}
    line.update(adjoint=None, visualisation=None, configs=None)
    bench.print_line(line)
    out = capsys.readouterr()
    assert out.err == "" and "legs" not in json.loads(out.out)
