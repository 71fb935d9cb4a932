"""bench.py's result is one JSON line on stdout that stays short whatever was
measured beside it; the side measurements go to stderr."""
import json

import bench


def test_side_measurements_stay_out_of_the_result_line(capsys):
    line = {"metric": bench.METRIC, "value": 1.0, "unit": bench.UNIT, "n_gpus": 1}
    trace = {"req_per_s": 15.1, "p50_s": 0.8, "p99_s": 2.9, "per_job": list(range(4000))}
    side = {"serving": {"capacity_req_per_s": 25.0, "configured_20_per_s": trace, "steady_state": trace},
            "studies": [[0.1234] * 64] * 64}
    bench.print_result(line, side)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and out.endswith("\n") and len(out) < 4000
    got = json.loads(out)
    assert {k: got[k] for k in line} == line
    assert got["serving"] == {"capacity_req_per_s": 25.0, "steady_state": {"req_per_s": 15.1, "p50_s": 0.8, "p99_s": 2.9}}
    assert json.loads(err) == {"side": side}


def test_without_side_measurements_only_the_line_is_printed(capsys):
    bench.print_result({"value": 2.0}, {})
    out, err = capsys.readouterr()
    assert json.loads(out) == {"value": 2.0} and err == ""
