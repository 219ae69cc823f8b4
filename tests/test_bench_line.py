"""The benchmark's line: one JSON object of bounded size, the rest in a file (no GPU)."""
import json
import os

import bench


def test_line_is_short_and_the_details_are_in_the_file(tmp_path):
    path = str(tmp_path / "sub" / "details.json")
    line = {"metric": bench.METRIC, "value": 1058123.123456789, "config": {"workload": bench.WORKLOAD_NAME, "note": "x" * 1500},
            "e2e": {"value": 1 / 3}, "us_per_step_blocks": {"n": 7, "median": 1 / 7, "pad": "y" * 600}}
    text = bench.emit(line, {"sweep": [{"us": 1 / 3}] * 500}, path)
    got = json.loads(text)
    assert "\n" not in text and len(text.encode()) <= bench.MAX_LINE
    assert got["value"] == 1058120.0 and got["e2e"]["value"] == 0.333333 and got["details"].endswith("details.json")
    with open(path) as f:
        whole = json.load(f)
    assert whole["value"] == line["value"] and len(whole["details"]["sweep"]) == 500
    long = dict(line, config={"note": "x" * 2200})
    got = json.loads(bench.emit(long, {}, path))
    assert "us_per_step_blocks" not in got and got["value"] == 1058120.0


def test_details_that_cannot_be_written_do_not_lose_the_line(tmp_path):
    blocked = tmp_path / "file"
    blocked.write_text("")
    got = json.loads(bench.emit({"value": 2.0}, {}, os.path.join(str(blocked), "details.json")))
    assert got == {"value": 2.0, "details": None}
