"""Offsets of a strip's rows within a plane, for planes up to the largest the
library takes (fewer than 2^31 elements): level row i sits at full-grid row
min(i * s, N - 1), and i * s * pitch of the last coarse row may reach 2^32.  The walk
over rows that the strip kernels use (csrc/mgr_rows.h) is compiled for the host and
compared with unbounded integers: every row of the level is exact, and what a strip
asks for before the first and past the last row stays within the plane."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_12764_gb300", "csrc")
SHAPES = [(100, 20_000_000), (10, 200_000_000), (1000, 2_100_000), (40_000, 53_000), (514, 2_097_152),
          (46_340, 46_340), (20, 100_000_000), (715_000_000, 3), (3, 715_000_000), (4, 536_870_911), (33, 17)]
MAX_STRIP = 16


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rows")
    src, lib = d / "rows.cpp", d / "rows.so"
    src.write_text('#include "mgr_rows.h"\n'
                   'extern "C" void walk(int first, int s, int N, int pitch, int units, int* coarse, int* fine, int* inner,'
                   ' int* above) {\n'
                   '  mgr::StripRows r(first, s, N, pitch);\n'
                   '  for (int pass = 0; pass < 2; ++pass, r.restart())\n'
                   '    for (int u = 0; u < units; r.next(u == 0), ++u) coarse[u] = r.coarse(), fine[u] = r.fine();\n'
                   '  for (int pass = 0; pass < 2; ++pass) {\n'
                   '    r.rewind();\n'
                   '    for (int u = 0; u < units; r.advance(), ++u) inner[u] = r.coarse(), above[u] = r.above();\n'
                   '  }\n'
                   '}\n')
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    walk = ctypes.CDLL(str(lib)).walk

    def rows(first, s, N, pitch, units):
        out = [(ctypes.c_int * units)() for _ in range(4)]
        walk(first, s, N, pitch, units, *out)
        return out

    return rows


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_row_offsets(rows, shape):
    N, pitch = shape
    assert N * pitch < 2 ** 31
    n, s = N, 1
    while n >= 3:
        m = n // 2 + 1
        for first in {*range(min(m, 40)), *range(max(m - 40, 0), m)}:
            units = MAX_STRIP + 2
            for step, length in ((1, n), (s, N)):  # a level's own values, the full grid
                coarse, fine, inner, above = rows(first, step, length, pitch, units)
                for u in range(units):
                    qc = first - 1 + u
                    if qc < m:
                        at = (2 * max(qc, 0), max(2 * qc - 1, 0))
                        want = tuple(min(i * step, length - 1) * pitch for i in at)
                        assert (coarse[u], fine[u]) == want, (n, step, first, u)
                        if qc >= 0:
                            assert inner[u] == want[0]
                        if qc >= 1:
                            assert above[u] == want[1]
                    assert all(0 <= v[u] <= (length - 1) * pitch for v in (coarse, fine, inner, above))
        n, s = m, 2 * s
