"""Blocks of an FP64 class launch, by the library's own plan compiled for the host: every link is in
one block, and a thread per link is taken exactly where its layers are the cheaper ones by the
measured times."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_09764_gb300", "csrc")
PROGRAM = """
#include <cstdio>
#include "vs_rows.cuh"
namespace vs { void count_launches(int) {} }
template <bool RECT>
void row(int n) {
    const vs::RowPlan<RECT> r = vs::row_plan<RECT>(n, 152);
    std::printf("%d %d %d %d %d %.6f %d\\n", n, RECT, r.n_whole, r.rest, r.sixes, r.us, vs::thread_layers<RECT>(n, 152));
}
int main() {
    for (int n = 64; n < 700000; n += n < 50000 ? 64 : 1088) { row<true>(n); row<false>(n); }
}
"""


def test_every_link_in_one_block(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "plan.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "plan")
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", exe, str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    picked = {}
    for line in subprocess.check_output([exe], text=True).splitlines():
        n, rect, whole, rest, sixes, us, thread = line.split()
        n, rect, whole, rest, sixes, us = int(n), int(rect), int(whole), int(rest), int(sixes), float(us)
        # whole blocks end at the links of the other blocks, or cover the last link themselves
        assert whole * 42 + rest == n if rest else (whole - 1) * 42 < n <= whole * 42
        if sixes:
            assert whole == 0 and rest == n
        layers = -(-n // 19456)
        own = 237.2 * layers + 9.6 if rect else 56.0 * layers + 5.8
        assert (thread == "1") == (own < us + (12 if rect else 8))
        picked[n, rect] = thread == "1"
    # the sizes whose times are in the table beside the rule
    for n, rect, want in ((64, 1, False), (1024, 0, False), (3456, 1, False), (10368, 0, False), (18432, 1, True),
                          (18432, 0, True), (32768, 1, False), (32768, 0, True), (36864, 1, True), (36864, 0, True)):
        assert picked[n, rect] == want, (n, rect)
