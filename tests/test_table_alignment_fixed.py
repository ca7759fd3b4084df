"""As test_table_alignment, for classes with the fixed-point form of NUMEROV_SPLIT: its tables lie behind the others, on
16-byte boundaries, and fit the class block, on odd and even grids."""
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
    static_assert(sizeof(FixPoint) == 16 && sizeof(FixObs) == 16, "entries are read as int4");
    int64_t base = 0;
    for (int N : {16, 17, 401, 1547, 4096, 32767, 32768})
        for (int ok : {0, 1}) {
            ClassDesc c{};
            c.N = N;
            c.tab_off = base;
            c.fix.num = 1;
            c.fix.ok = ok;
            const int64_t at[] = {tab_xff(c), tab_fxp(c), tab_fob(c), tab_fnw(c), base + tab_doubles(c)};
            const int64_t len[] = {2, 2, 2, 6};   // doubles per point; fnw: three int4
            for (int k = 0; k < 4; ++k)
                if (at[k] % 2 != 0 || at[k] + len[k] * N > at[k + 1]) return 1 + k;
            base += tab_doubles(c);
            if (base % 2) return 20;
        }
    return 0;
}
"""


def test_fixed_point_tables_are_aligned(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-I" + CSRC, "-I" + INCLUDE, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
