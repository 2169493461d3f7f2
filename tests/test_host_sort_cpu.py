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


FAILING = r"""
#include <cstdio>
#include <new>
#include "host_sort.h"
static int made, joined, fail_at, kind;
struct Thread {
    bool joinable = true;
    template <class F> Thread(F f, int t) {
        if (t == fail_at) {
            if (kind == 0) throw std::bad_alloc();
            throw std::system_error(std::make_error_code(std::errc::resource_unavailable_try_again));
        }
        ++made;
        f(t);
    }
    Thread(Thread &&o) : joinable(o.joinable) { o.joinable = false; }
    ~Thread() { if (joinable) std::terminate(); }
    void join() { joinable = false; ++joined; }
};
int main() {
    for (kind = 0; kind < 2; ++kind)
        for (fail_at = 1; fail_at <= 6; ++fail_at) {
            made = joined = 0;
            int seen[6] = {};
            fstat::parallel_for_threads<Thread>(6, [&](int t) { ++seen[t]; });
            int once = 0;
            for (int v : seen) once += v == 1;
            printf("%d %d %d\n", made, joined, once);
        }
}
"""


def test_threads_that_cannot_be_made(tmp_path):
    """Whatever the creation of a thread throws, the threads made before are joined and every
    slice of the loop has run once."""
    v = [int(x) for x in _run(tmp_path, FAILING.replace("#include <new>", "#include <new>\n#include <system_error>"))]
    assert v == 2 * [x for f in range(1, 7) for x in (f - 1 if f < 6 else 5, f - 1 if f < 6 else 5, 6)]
