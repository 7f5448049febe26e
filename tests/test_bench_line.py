"""The benchmark's result: one line on stdout, short enough that the end of an output holds all of it."""
import json

import bench


def test_the_result_is_one_short_line_and_the_tables_go_to_stderr(capsys):
    line = {"metric": "m", "value": 1234.56789, "config": {"workload": "w", "l2": "ring of buffers larger than L2" * 4},
            "e2e": {"value": 1.0, "unit": "TOPS", "h2d_bytes_per_step": 16777216, "d2h_bytes_per_step": 16777216, "api": "a" * 900},
            "clocks": {"sm_mhz": 1965.0, "reasons": []}, "roofline": {"frac": 2.0 / 3.0, "peak_source": "p" * 1500}}
    tables = {"per_workload": {"w%d" % i: {"ms": 0.1} for i in range(200)}}
    bench.print_line(line, tables)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) <= bench.LINE_LIMIT + 1
    got = json.loads(out)
    assert got["value"] == 1234.57 and got["e2e"]["h2d_bytes_per_step"] == 16777216 and got["e2e"]["unit"] == "TOPS"
    assert got["config"] == line["config"] and got["clocks"] == line["clocks"] and "per_workload" not in got
    full = json.loads(err)
    assert full["per_workload"] == tables["per_workload"] and full["roofline"]["peak_source"] == "p" * 1500


def test_a_short_line_without_tables_leaves_stderr_alone(capsys):
    bench.print_line({"metric": "m", "value": 1.0}, {})
    out, err = capsys.readouterr()
    assert json.loads(out) == {"metric": "m", "value": 1.0} and err == ""
