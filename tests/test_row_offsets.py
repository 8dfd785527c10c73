"""Offsets of a level's rows within a plane, for planes up to the largest the
library takes (fewer than 2^31 elements): level row i sits at full-grid row
min(i * 2^k, N - 1), so the product of row index and pitch fits in 32 bits only
once the row is clamped.  The expression the strip kernels use
(csrc/mgr_rows.h) is compiled for the host and compared with unbounded integers
over every row a strip may ask for: from the two before the grid to a strip's
height past its end."""
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
def offset(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("rows")
    src, lib = d / "rows.cpp", d / "rows.so"
    src.write_text('#include "mgr_rows.h"\n'
                   'extern "C" int offset(int i, int n, int s, int N, int pitch) {\n'
                   '  return mgr::level_row_offset(i, n, s, N, pitch);\n}\n')
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib)).offset


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_row_offsets(offset, shape):
    N, pitch = shape
    assert N * pitch < 2 ** 31
    n, s = N, 1
    while n >= 3:
        for i in {*range(-2, min(n + 2 * MAX_STRIP, 70)), *range(max(n - 70, -2), n + 2 * MAX_STRIP)}:
            # compact rows (a level's own values) and full-grid rows
            assert offset(i, n, 1, n, pitch) == min(max(i, 0), n - 1) * pitch, (n, i)
            assert offset(i, n, s, N, pitch) == min(max(i, 0) * s, N - 1) * pitch, (n, s, i)
        n, s = n // 2 + 1, 2 * s
        if n == 2:
            break
