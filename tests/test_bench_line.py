"""The benchmark's result: one line on stdout, short enough that the end of an output holds all of it."""
import json

import bench
import csrc_util
from paper_2511_22316_b200 import workloads as wl


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


def test_a_captured_traffic_is_printed_beside_its_own_kernel_only():
    for (step, name), (kernel, nbytes) in bench.NCU_TRAFFIC.items():
        assert bench.ncu_traffic(step, name, kernel) == nbytes and bench.ncu_traffic(step, name, "another") is None
        w = wl.by_name(name)
        takes = {"gemm": bench.gemm_kernel_name(w), "wo_gemm": bench.wo_gemm_kernel_name(w.M, w.N, w.K)}.get(
            step, bench.rotate_kernel_name(w, step == "rotate_quant_st"))
        assert kernel == takes, (step, name)
    assert bench.ncu_traffic("gemm", "no such workload", "w4a4_gemv_kernel") is None


def test_kernel_names_follow_the_lines_of_the_stream_kernels():
    shapes = [(M, N, K) for M in (1, 2, 3, 8, 9) for N in (126, 128, 131, 1024, 1032, 4096, 4738, 7104, 7106, 8192, 8200, 9472, 9480)
              for K in (224, 256, 512, 1056, 2048, 2080, 3072, 4096, 4112, 7168, 7200, 12288, 12416, 16384, 16512, 28672, 32800)]
    for (M, N, K), (w4a4, wo) in zip(shapes, csrc_util.stream_takes(shapes), strict=True):
        assert bench.stream_kernel_takes(M, N, K) == w4a4, (M, N, K)
        assert (bench.wo_gemm_kernel_name(M, N, K) == "wo_gemm_stream_kernel") == wo, (M, N, K)
