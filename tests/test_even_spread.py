"""Shared memory that a dependent launch of less than a full chip asks for, by the library's own
function compiled for the host: as many of its blocks fit an SM as an even spread gives, and what the
kernel needs is never cut."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_09764_gb300", "csrc")
SMS, ALL, RESERVED, MOST = 152, 233472, 1024, 232448
PROGRAM = """
#include <cstdio>
#include "vs_stout.cuh"
namespace vs { void count_launches(int) {} }
int main() {
    for (int smem : {36864, 55296})
        for (int per : {0, 3, 4})
            for (int b = 1; b <= 800; ++b)
                std::printf("%d %d %d %d\\n", smem, per, b, vs::even_smem(b, smem, per, 152, 233472, 1024, 232448));
}
"""


def test_blocks_per_sm(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "spread.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "spread")
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", exe, str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    for line in subprocess.check_output([exe], text=True).splitlines():
        smem, per, blocks, got = map(int, line.split())
        even = -(-blocks // SMS)
        if even >= per:
            assert got == smem
            continue
        assert smem <= got <= MOST
        assert ALL // (got + RESERVED) == even
