"""The class tables' offsets: every table that the kernels read as double2 or float4 starts on a 16-byte
boundary and holds its elements, for odd and even grids (compiled from the library's own header)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_04115_gb300", "csrc")
INCLUDE = os.path.join(os.path.dirname(os.path.dirname(CSRC)), "include")
PROGRAM = """
#include "tdse_internal.h"
using namespace tdse;
int main() {
    int64_t base = 0;
    for (int N : {16, 17, 401, 1547, 4096, (1 << 20) - 1}) {
        ClassDesc c{};
        c.N = N;
        c.tab_off = base;
        c.fix.ok = 1;
        const int64_t at[] = {tab_ab(c), tab_xv(c), tab_mk(c), tab_nw(c), tab_nl(c), tab_nc(c),
                              tab_nf(c), tab_fx(c), tab_vv(c), tab_af(c), tab_xff(c), tab_fxp(c), tab_fob(c), base + tab_doubles(c)};
        const int64_t len[] = {2, 2, 1, 2, 2, 2, 3, 2, 1, 1, 2, 2, 2};   // doubles per point
        for (int k = 0; k < 13; ++k)
            if (at[k] % 2 != 0 || at[k] + len[k] * N > at[k + 1]) return 1 + k;
        base += tab_doubles(c);
        if (base % 2) return 20;
        c.fix.ok = 0;   // classes without the fixed-point form end before its tables
        if (tab_doubles(c) > tab_fxp(c) - c.tab_off) return 21;
    }
    return 0;
}
"""


def test_tables_are_aligned_for_vector_loads(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-I" + CSRC, "-I" + INCLUDE, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
