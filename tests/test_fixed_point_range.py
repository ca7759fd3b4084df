"""The range of the fixed-point FULL_CN sweep that the header states (include/tdse.h, TDSE_FP64), from the library's own
rule (csrc/tdse_internal.h, class_fix)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC, INCLUDE = os.path.join(ROOT, "paper_2507_04115_gb300", "csrc"), os.path.join(ROOT, "include")
PROGRAM = """
#include "tdse_internal.h"
#include <cstdio>
#include <cstdlib>
using namespace tdse;
int main(int, char** v) {
    ClassDesc c{};
    c.N = atoi(v[1]);
    c.dx = atof(v[2]);
    c.a = 1.19;
    c.Z = 1.0;
    const FixClass f = class_fix(c, atof(v[3]));
    printf("%d %.17g\\n", f.ok, f.E_lim);
    return 0;
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("range")
    (d / "t.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-I" + CSRC, "-I" + INCLUDE, "-o", str(d / "t"), str(d / "t.cu")], check=True)

    def run(N, dx, dt):
        ok, lim = subprocess.run([str(d / "t"), str(N), str(dx), str(dt)], capture_output=True, text=True, check=True).stdout.split()
        return bool(int(ok)), float(lim)
    return run


def test_field_limit_as_stated(rule):
    for N, dx, dt, lim in ((4096, 0.15, 0.02, 0.94), (8192, 0.2, 0.02, 0.20), (16384, 0.2, 0.02, 0.10), (32768, 0.2, 0.02, 0.05)):
        ok, e = rule(N, dx, dt)
        assert ok and abs(e - lim) < 0.006 and abs(e * N * dx ** 3 - 13.0) < 0.2
    text = re.sub(r"\s+", " ", open(os.path.join(INCLUDE, "tdse.h")).read())
    assert "13 / (N dx^3) (0.94 a.u. at N = 4096, dx = 0.15; 0.20, 0.10 and 0.05 at dx = 0.2 and N = 8192, 16384 and 32768)" in text


def test_grids_outside_as_stated(rule):
    for N, dx, dt, ok in ((4096, 0.1, 0.02, False), (4096, 0.15, 0.05, False), (4096, 0.2, 0.01, False), (32769, 0.2, 0.02, False),
                          (4096, 0.2, 0.02, True), (4096, 0.2, 0.05, True), (32768, 0.15, 0.02, True), (4096, 0.2, 0.0561, False),
                          (4096, 0.2, 0.01143, False), (4096, 0.2, 0.01145, True), (4096, 0.2, 0.05599, True)):
        assert rule(N, dx, dt)[0] == ok, (N, dx, dt)
