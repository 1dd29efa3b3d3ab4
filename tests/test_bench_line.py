"""bench.py's result line: one JSON line that stays short whatever was measured besides, the rest on a line of its own."""
import io
import json

import bench


def test_result_line_is_short_and_details_are_apart():
    stats = {"median": [1.0 / 3.0] * 4, "frac_le_1e-8": [2.0 / 3.0] * 4}
    extra = {"order8_mixed_vs_fp64": {p: {"ms": 1.23456789, "mnodes_per_s": 4.5, "refine_steps": [0] * 8} for p in ("fp64", "mixed", "mixed_tc")},
             "accuracy_vs_oracle": {"orders": {str(k): {"ops": ["dx"], "sample": {"nodes": 512, "fp64": stats, "mixed": stats}} for k in range(2, 9)}},
             "filler": [[1.0 / 7.0] * 100] * 100}
    line = {"metric": bench.METRIC, "value": 4.0 / 3.0, "e2e": {"value": 1.0}, "extra": extra}
    out, err = io.StringIO(), io.StringIO()
    bench.report(line, out, err)
    text = out.getvalue()
    assert text.count("\n") == 1 and len(text) < 4000
    got = json.loads(text)
    assert got["value"] == 1.33333 and got["metric"] == bench.METRIC and got["e2e"] == {"value": 1.0} and "extra" not in got
    assert got["mixed_vs_fp64"]["order8"]["mixed_tc"] == {"ms": 1.23457, "mnodes_per_s": 4.5}
    assert got["order8_frac_le_1e-8"] == {"sample": {"fp64": [0.666667] * 4, "mixed": [0.666667] * 4}}
    details = err.getvalue()
    assert details.startswith("bench details: ") and details.count("\n") == 1
    assert set(json.loads(details[len("bench details: "):])) == set(extra)
    assert "extra" in line  # the caller's own line is left as it was
