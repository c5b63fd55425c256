"""Threads of a class launch, by the library's own functions compiled for the host: every link of the
class is taken by one thread, whether warps take sites in order or whole runs, and whole runs (18
reals, rows of 20) are taken only where their further blocks add at most one layer over the SMs to
every fourteen."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_09764_gb300", "csrc")
SMS, BLOCK = 152, 128
LINKS = [64, 320, 19200, 19456, 19520, 35840, 38400, 38912, 40320, 57600, 64000, 76800, 80000, 96000, 259200, 320000,
         599040]
PROGRAM = """
#include <cstdio>
#include <vector>
#include "vs_stout.cuh"
namespace vs { void count_launches(int) {} }
template <int NC>
void row(int lx, int n, bool one_class) {
    const int dims[4] = {lx, 4, 4, 4};
    const bool runs = one_class && vs::whole_runs<NC>(vs::make_geo(dims), n, 152);
    const int threads = runs ? vs::whole_run_threads(n) : n;
    const int colour = one_class ? (runs ? 3 | vs::kRuns : 3) : -1;
    std::vector<int> taken(n, 0);
    bool once = threads >= n;
    for (int k = 0; k < (threads + 127) / 128 * 128; ++k) {
        const int t = vs::class_thread<NC>(colour, k, n);
        if (t >= 0 && t < n) once &= ++taken[t] == 1;
    }
    for (int c : taken) once &= c == 1;
    std::printf("%%d %%d %%d %%d %%d %%d %%d\\n", NC, lx, n, one_class, runs, threads, once);
}
int main() {
    for (int n : {%s})
        for (int lx : {12, 20, 24, 28})
            for (bool one_class : {false, true}) { row<18>(lx, n, one_class); row<12>(lx, n, one_class); }
}
""" % ", ".join(map(str, LINKS))


def test_every_link_once_and_runs_where_they_pay(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "runs.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "runs")
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-o", exe, str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    seen = set()
    for line in subprocess.check_output([exe], text=True).splitlines():
        nc, lx, n, one_class, runs, threads, once = map(int, line.split())
        assert once
        whole = -(-n // 30) * 32
        layers = [-(-t // (BLOCK * SMS)) for t in (n, whole)]
        pays = layers[1] - layers[0] <= layers[0] // 14
        assert runs == (nc == 18 and lx == 20 and one_class == 1 and pays)
        assert threads == (whole if runs else n)
        seen.add((n, runs))
    assert (38400, 1) not in seen and (35840, 1) in seen and (80000, 1) in seen
