"""Byte offset of a link in its direction for every storage, by the library's own functions compiled
for the host, against the layout's formula in exact integers, up to the largest field of each storage:
2^30 positions, or 64 GiB per direction (18 i passes 2^31 at 119,304,648 positions, 12 i at
178,956,971)."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_09764_gb300", "csrc")
POSITIONS = [0, 15, 16, 31, 255, 119304639, 119304648, 134217727, 178956971, 268435455, 477218303, 477218304,
             2 ** 29 + 5, 954436863, 954436864, 2 ** 30 - 1]
PROGRAM = """
#include <cstdio>
#include "vs_device.cuh"
int main() {
    const int at[] = {%s};
    const char *z = reinterpret_cast<const char *>(1ull << 40);
    const float *f = reinterpret_cast<const float *>(z);
    for (int i : at) {
        const void *p[4] = {vs::blk_float4<18>(f, i), vs::blk_float4<12>(f, i), vs::blk_float2(f, i),
                            vs::blk_double2(reinterpret_cast<const double *>(z), i)};
        for (const void *q : p) std::printf("%%lld ", (long long)(static_cast<const char *>(q) - z));
        const long long P = (i / 256 + 1) * 256ll;
        std::printf("%%d %%d %%d\\n", vs::links_fit(P, 72), vs::links_fit(P, 48), vs::links_fit(P, 144));
    }
}
""" % ", ".join(map(str, POSITIONS))


def test_offsets_up_to_the_largest_field(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "offsets.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "offsets")
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", exe, str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    rows = [tuple(map(int, line.split())) for line in subprocess.check_output([exe], text=True).splitlines()]
    for i, (f18, f12, f18_last, d18, fit72, fit48, fit144) in zip(POSITIONS, rows):
        b, e = divmod(i, 16)      # block of 16 links, element
        P = (i // 256 + 1) * 256  # the smallest plane that holds position i
        assert (fit72, fit48, fit144) == tuple(int(P * n <= 2 ** 36) for n in (72, 48, 144))
        if fit72:
            assert (f18, f18_last) == (1152 * b + 16 * e, 1152 * b + 1024 + 8 * e)
        if fit48:
            assert f12 == 768 * b + 16 * e
        if fit144:
            assert d18 == 2304 * b + 16 * e
    # every storage reaches the positions at which an int offset in reals would wrap
    assert all(r[4] for r in rows[:11]) and all(r[5] for r in rows) and all(r[6] for r in rows[:10])
