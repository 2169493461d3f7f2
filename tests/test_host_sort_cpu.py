"""The host sort of candidate records (csrc/host_sort.h), compiled for the host: every record
count around the run boundaries of one to seven threads, narrow and wide keys, against a
stable comparison sort by (cell, bin)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1410_3677_gb300", "csrc")

PROG = r"""
#include <cstdio>
#include <random>
#include "host_sort.h"
struct Rec { uint32_t cell, bin; double F; };
int main() {
    std::mt19937_64 g(7);
    int bad = 0, runs = 0;
    for (int nt : {1, 2, 3, 7})
        for (long n : {0L, 1L, 2L, 63L, 64L, 65L, 1000L, 65537L, 200001L})
            for (int cb : {0, 1, 12, 32})
                for (int bb : {1, 7, 13, 20}) {
                    const uint32_t cell0 = cb == 32 ? 0 : 1000, bin0 = 5;
                    std::vector<Rec> a(n), tmp(n);
                    for (long i = 0; i < n; ++i)
                        a[i] = {cell0 + (uint32_t)(g() & ((uint64_t(1) << cb) - 1)), bin0 + (uint32_t)(g() & ((1u << bb) - 1)), (double)i};
                    auto b = a;
                    std::stable_sort(b.begin(), b.end(), [](const Rec &x, const Rec &y) {
                        return x.cell != y.cell ? x.cell < y.cell : x.bin < y.bin; });
                    fstat::sort_records(a.data(), tmp.data(), n, cell0, bin0, bb, cb + bb, nt);
                    ++runs;
                    for (long i = 0; i < n; ++i)
                        if (a[i].cell != b[i].cell || a[i].bin != b[i].bin || (n >= 64 && a[i].F != b[i].F)) { ++bad; break; }
                }
    printf("%d %d\n", runs, bad);
}
"""


def _run(tmp_path, prog):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    src = tmp_path / "p.cpp"
    src.write_text(prog)
    exe = str(tmp_path / "p")
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", f"-I{CSRC}", str(src), "-o", exe], check=True,
                   capture_output=True)
    return subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()


def test_host_sort_matches_a_stable_sort(tmp_path):
    runs, bad = _run(tmp_path, PROG)
    assert int(runs) == 4 * 9 * 4 * 4 and int(bad) == 0
