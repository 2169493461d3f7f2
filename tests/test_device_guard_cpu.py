"""The guard that makes a plan's calls run on the plan's device (csrc/device_guard.h), compiled
for the host over a counted stand-in of the get and set calls, and its place in every call
that takes a plan."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1410_3677_gb300", "csrc")

PROG = r"""
#include <cstdio>
#include "device_guard.h"
struct Api {
    static int current, sets, fail;
    static bool get(int *d) { *d = current; return fail != 1; }
    static bool set(int d) { if (fail == 2) return false; ++sets; current = d; return true; }
};
int Api::current, Api::sets, Api::fail;
static void run(int current, int device, int fail) {
    Api::current = current; Api::sets = 0; Api::fail = fail;
    int inside, ok;
    {
        fstat::DeviceGuard<Api> g(device);
        inside = Api::current;
        ok = g.ok();
    }
    printf("%d %d %d %d\n", inside, ok, Api::current, Api::sets);
}
int main() {
    run(0, 1, 0);    // a thread on device 0, a plan on device 1
    run(1, 1, 0);    // the plan's device already: no call
    run(2, -1, 0);   // no device known
    run(0, 1, 1);    // the current device cannot be read
    run(0, 1, 2);    // it cannot be changed: nothing to restore
}
"""


def test_guard_changes_and_restores_the_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    src = tmp_path / "g.cpp"
    src.write_text(PROG)
    exe = str(tmp_path / "g")
    subprocess.run([cxx, "-O1", "-std=c++17", f"-I{CSRC}", str(src), "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")[:-1]
    assert out == ["1 1 0 2", "1 1 1 0", "2 1 2 0", "0 0 0 0", "0 0 0 0"]


def test_every_call_on_a_plan_is_guarded():
    """Calls that work on a mutable plan go through guarded(), which holds the guard before the
    call's body, or hold it themselves."""
    txt = open(os.path.join(CSRC, "api.cu")).read()
    body = txt[txt.index("fstat_status guarded("):]
    assert body.index("DeviceGuard<CudaDevice> on_device(p->device)") < body.index("return f();")
    for m in re.finditer(r"^(?:fstat_status|void) (fstat_\w+)\(fstat_plan \*p[,)][^{]*\{\n(.*)\n(.*)\n", txt, re.M):
        name, first, second = m.groups()
        assert "return guarded(p, " in first or "DeviceGuard<CudaDevice> on_device(p->device)" in second, name
    assert len(re.findall(r"return guarded\(p, ", txt)) >= 6


def test_no_process_wide_state_stands_for_a_device():
    """A kernel's shared-memory limit and the number of its CTAs that fit belong to a device: no
    function-local flag or count of the process decides about them."""
    for f in sorted(os.listdir(CSRC)):
        txt = open(os.path.join(CSRC, f)).read()
        assert not re.findall(r"\n +static (?:bool|int|size_t) \w+(?:\[[^\]]*\])? *[={;][^\n]*", txt), f
