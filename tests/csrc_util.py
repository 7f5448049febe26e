"""Pieces of the CUDA sources compiled for the host: layouts and dispatch rules are checked as they stand there."""
import os
import re
import subprocess
import tempfile

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_22316_b200", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def block(text, head):
    """From `head` to the closing brace, at the start of a line, of what it opens (a struct or a function)."""
    start = text.index(head)
    end = text.index("\n}", start) + 2
    return text[start:end] + (";" if text[end:end + 1] == ";" else "")


def lines(text, pattern):
    return "\n".join(re.findall(pattern, text, re.M))


def run(code, *args):
    """Compiles `code` (a program; CUDA's qualifiers mean nothing here) and returns the lines it prints, split."""
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "p.cpp"), os.path.join(d, "p")
        with open(src, "w") as f:
            f.write("#include <algorithm>\n#include <cmath>\n#include <cstdint>\n#include <cstdio>\n#include <cstdlib>\n"
                    "#define __host__\n#define __device__\n#define __forceinline__ inline\n" + code)
        subprocess.run(["g++", "-std=c++17", "-o", exe, src], check=True)
        out = subprocess.run([exe] + [str(a) for a in args], check=True, capture_output=True, text=True).stdout
    return [line.split() for line in out.splitlines()]


def wo_pair_widths(shapes, pairs=74):
    """The token width that the weight-only CTA-pair product takes for each (M, N), on `pairs` CTA pairs."""
    wo = source("sq_gemm_wo.cu")
    code = (lines(wo, r"^constexpr int WP_TILE_STEP.*$") + "\n" + block(wo, "int wo_pair_tile_m(")
            + "\nint main(int n, char** v) { for (int i = 1; i + 1 < n; i += 2)"
              " printf(\"%d\\n\", wo_pair_tile_m(atoi(v[i]), atoi(v[i + 1]), PAIRS)); }")
    return [int(row[0]) for row in run(code.replace("PAIRS", str(pairs)), *[v for s in shapes for v in s])]


def stream_takes(shapes):
    """For each (M, N, K) whether the stream kernels take the W4A4 and the weight-only product, on 148 SMs."""
    src = source("sq_gemm_stream.cu")
    rows = run(lines(src, r"^constexpr int SM_.*$") + "\nint sm_count() { return 148; }\n"
               + block(source("sq_gemm_decode.cu"), "bool gemm_decode_supported(") + block(source("sq_gemv.cu"), "bool gemv_supported(")
               + block(src, "static bool stream_yields(") + block(src, "bool w4a4_stream_supported(")
               + block(src, "bool wo_stream_supported(") + """
int main(int n, char** v) {
  for (int i = 1; i + 2 < n; i += 3) {
    const int M = atoi(v[i]), N = atoi(v[i + 1]), K = atoi(v[i + 2]);
    printf("%d %d\\n", w4a4_stream_supported(M, N, K), wo_stream_supported(M, N, K));
  }
}""", *(v for s in shapes for v in s))
    return [(row[0] == "1", row[1] == "1") for row in rows]
