"""What of the benchmark's result goes into its one line on stdout."""
import json

import bench


def _line(**tables):
    return {"metric": bench.METRIC, "value": 1.0, "e2e": {"value": 0.5}, **tables}


def test_the_line_of_a_full_run_is_short():
    rows = [{"config": "row%d" % k, "gemm_loss": k / 100, "matches_oracle": True} for k in range(12)]
    tables = {"large_messages": {"all_match_oracle": True, "rows": rows * 50}, "gemm_loss_matched": {"rows": rows}, "extras": {"x": list(range(9999))}}
    line = _line(**tables)
    assert bench.split_tables(line, "auto") == tables
    assert line == _line(gemm_loss={r["config"]: r["gemm_loss"] for r in rows}, large_messages_match_oracle=True) and len(json.dumps(line)) < 1000


def test_tables_stay_in_the_line_when_asked_for_or_without_extras():
    for where, tables in (("auto", {"large_messages": {"rows": []}}), ("line", {"extras": {}, "large_messages": {"rows": []}})):
        line = _line(**tables)
        assert bench.split_tables(line, where) == {} and line == _line(**tables)
    line = _line(gemm_loss_matched={"rows": []})
    assert list(bench.split_tables(line, "stderr")) == ["gemm_loss_matched"] and line == _line(gemm_loss={})
