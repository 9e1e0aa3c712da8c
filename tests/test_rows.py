"""Row numbers of a segment (csrc/rows.cuh) against 64-bit arithmetic, near 2^31 rows and on grids of a few: the rows a warp reads,
which of them lie in the grid, and the periodic wrap."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1107_4650_gb300", "csrc")

HARNESS = r'''
#include "rows.cuh"
#include <initializer_list>
#include <stdio.h>
int main() {
    long bad = 0, seen = 0;
    const int64_t top = 0x7fffffff;
    for (int64_t nr : {(int64_t)1, (int64_t)2, (int64_t)3, (int64_t)17, (int64_t)1000, top / 2, dirac::kMaxSegRows, dirac::kMaxSegRows + 3, top - 70, top - 3, top - 1, top})
        for (int64_t h : {(int64_t)1, (int64_t)2, (int64_t)16, (int64_t)61, (int64_t)4096, dirac::kMaxSegRows}) {
            const int64_t segs = (nr + h - 1) / h;
            for (int64_t seg : {(int64_t)0, (int64_t)1, segs / 2, segs - 2, segs - 1}) {
                if (seg < 0 || seg >= segs) continue;
                const dirac::SegRows s = dirac::seg_rows(seg, h, nr);
                bad += s.row0 != seg * h || s.end != (h < nr - seg * h ? h : nr - seg * h);
                for (int edge = 0; edge < 2; ++edge)
                    for (int d = -12; d <= 12; ++d) {  // four levels and four slots beyond either end, and rows inside
                        const int64_t wide = (edge ? s.end : 0) + (int64_t)d;
                        if (wide < -8 || wide > s.end + 8) continue;
                        const int r = (int)wide;
                        const int64_t g = s.row0 + r;
                        bad += dirac::row_in_grid((uint32_t)s.row0, r, (uint32_t)nr) != (g >= 0 && g < nr) || (r < s.top) != (g < nr);
                        if (g >= -8 && g <= nr + 8) bad += dirac::wrap_row((uint32_t)s.row0, r, (uint32_t)nr) != (uint64_t)(((g % nr) + nr) % nr);
                        ++seen;
                    }
            }
        }
    printf("%ld of %ld\n", bad, seen);
    return bad != 0 || seen < 1000;
}
'''


def test_rows_of_segments(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-O1", "-fsanitize=signed-integer-overflow", "-fno-sanitize-recover", "-I", CSRC, str(src), "-o",
                    str(tmp_path / "t")], check=True)
    out = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
