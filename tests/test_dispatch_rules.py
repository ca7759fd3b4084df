"""The host rules of the batch-free entry points (csrc/tdse_rules.h), compiled for the host."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_04115_gb300", "csrc")


def _run(tmp_path, body):
    if shutil.which("g++") is None:
        pytest.skip("g++ not found")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "tdse_rules.h"\n#include <cstdio>\nusing namespace tdse;\nint main() {\n%s\nreturn 0; }\n' % body)
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)


def test_field_passes_are_bounded(tmp_path):
    """The scratch of a resampling pass stays within 5/4 of its room and the twiddles, however many rows and outputs
    there are, down to a pass of one row and one output."""
    _run(tmp_path, """
    const size_t MB = size_t(1) << 20;
    for (size_t room = 512 * MB; room >= MB / 2; room /= 8)
        for (int M : {2, 3, 100, 2400, 8191, 8192})
            for (int64_t rows : {int64_t(1), int64_t(7), int64_t(100000), int64_t(1) << 31})
                for (int64_t n : {int64_t(1), int64_t(55160), int64_t(1000000000), int64_t(1) << 40}) {
                    const FieldPlan p = resample_field_plan(rows, M, n, room);
                    if (p.rows < 1 || p.rows > rows || p.rows > 65535 || p.outputs < (p.direct ? 0 : 1) || p.outputs > n) return 1;
                    const size_t least = 16 * (size_t)(M / 2 + 1) + 8 * (size_t)field_nodes(M) + 132;   // one row, one output
                    const size_t twiddles = 16 * (size_t)(M + field_nodes(M) / 2);
                    if (p.bytes > room + room / 4 + least + twiddles) return 2;
                    if (!p.direct && p.bytes < (size_t)p.rows * 8 * field_nodes(M) + (size_t)p.outputs * 132 + twiddles) return 3;
                    if (p.direct && p.bytes < (size_t)p.rows * 16 * (M / 2 + 1)) return 3;
                }
    const FieldPlan p = resample_field_plan(256, 2400, 55160, 512 * MB);   // a workload's call: one pass
    if (p.rows != 256 || p.outputs != 55160) return 4;
    """)


def test_field_route_follows_the_measured_calls(tmp_path):
    """(rows, M, outputs) measured at least 10 % apart: the quicker route."""
    _run(tmp_path, """
    struct { int64_t rows; int M; int64_t n; bool direct; } c[] = {
        {1, 2, 1000, true}, {32, 2, 1000, true}, {1, 600, 1000, false}, {1, 2400, 1000, false}, {1, 300, 12000, true},
        {32, 100, 12000, false}, {4, 600, 12000, false}, {8, 100, 55160, true}, {16, 100, 55160, false}, {8, 300, 55160, false},
        {1, 100, 400000, true}, {8, 100, 400000, true}, {32, 30, 400000, false}, {1, 1200, 400000, true}, {2, 1200, 400000, false},
        {1, 2400, 55160, false}, {256, 2400, 55160, false}, {1, 8192, 1000000, false}};
    for (auto& k : c)
        if (field_direct(k.rows, k.M, k.n) != k.direct) { printf("%d %d\\n", (int)k.rows, k.M); return 1; }
    """)


def test_j0_table_where_it_pays(tmp_path):
    """(source points, frequencies, radii, largest argument) measured more than 15 % apart on 152 SMs: the quicker
    route; and no table for arguments that overflow."""
    _run(tmp_path, """
    struct { int nr, nz, nw, no; double x; bool table; } c[] = {
        {1, 1, 8, 16, 3, false}, {4, 4, 40, 64, 20, false}, {16, 16, 40, 64, 20, true}, {32, 32, 20, 64, 3, true},
        {32, 32, 340, 256, 3, true}, {8, 8, 340, 512, 20, true}, {8, 8, 40, 64, 500, false}, {16, 16, 40, 64, 500, true},
        {4, 4, 340, 512, 500, false}, {16, 16, 340, 128, 1500, true}, {4, 4, 340, 512, 1500, false}, {16, 16, 40, 64, 4000, false},
        {16, 16, 340, 128, 4000, false}, {32, 32, 100, 256, 4000, true}, {8, 8, 340, 512, 4000, false},
        {32, 32, 20, 64, 20000, false}, {32, 32, 340, 256, 20000, true}};
    for (auto& k : c) {
        const int n = j0_table_nodes(k.x, k.nr, k.nz, k.nw, k.no, 152);
        if ((n > 0) != k.table) { printf("%d %d %d %g: %d\\n", k.nr, k.nw, k.no, k.x, n); return 1; }
        if (n > kJ0MaxNodes || (n > 0 && n < kJ0MaxNodes && n < 4 * k.x + 2)) return 2;
    }
    const double inf = 1e308 * 10;
    if (j0_table_nodes(inf, 1024, 1024, 340, 256, 152) || j0_table_nodes(inf - inf, 1024, 1024, 340, 256, 152)) return 3;
    if (j0_table_nodes(0.0, 1024, 1024, 340, 256, 152) > 3 || j0_table_nodes(1e300, 2048, 1024, 65535, 256, 152) > kJ0MaxNodes) return 4;
    """)


def test_moments_where_they_pay(tmp_path):
    """(rows, samples, bins from 0) measured more than 8 % apart on 152 SMs: the quicker route of the power spectrum."""
    _run(tmp_path, """
    struct { int64_t rows, L, nw; bool moments; } c[] = {
        {1, 512, 32, false}, {4, 512, 60, false}, {64, 512, 60, false}, {256, 512, 60, false}, {4, 1000, 60, false},
        {64, 1000, 32, false}, {256, 1000, 32, true}, {1, 2000, 32, true}, {4, 2000, 60, true}, {4, 2000, 120, false},
        {256, 2000, 120, true}, {1, 4000, 400, true}, {4, 4000, 400, false}, {16, 4000, 400, false}, {64, 4000, 400, true},
        {16, 4000, 120, true}, {4, 8000, 400, true}, {1, 20000, 32, true}, {256, 20000, 400, true}, {512, 55160, 400, true}};
    for (auto& k : c) {
        int B = 0, P = 0;
        const bool m = dft_plan(k.L, 2.0 * 3.141592653589793 * (k.nw - 1) / k.L, k.nw, k.rows, 152, &B, &P);
        if (m != k.moments) { printf("%d %d %d: %d\\n", (int)k.rows, (int)k.L, (int)k.nw, (int)m); return 1; }
        if (m != (B > 0)) return 2;
    }
    """)
