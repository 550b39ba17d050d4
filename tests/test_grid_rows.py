"""The grid rows of a view's footprint for poses far outside the map, on the host: the header the kernels include, compiled with
the undefined-behaviour checks on."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <climits>
#include <cstdio>
#include "pic_rows.h"
int main() {
    const float far[] = {-INFINITY, -3e38f, -1e12f, -2147483904.f, -2147483648.f, -33.f, -1.f, 0.f, 1.f, 31.f, 32.f, 53.f, 54.f, 1023.f,
                         2147483520.f, 2147483648.f, 1e12f, 3e38f, INFINITY, NAN};
    const unsigned rows[] = {1, 31, 32, 33, 54, 1024};
    for (unsigned ny : rows)
        for (float f0 : far)
            for (float f1 : far) {
                if (f0 > f1) continue;
                int lo = INT_MIN, hi = INT_MIN;
                pic::clamp_rows(f0, f1, ny, lo, hi);
                if (lo < 0 || lo > (int)ny || hi < -1 || hi > (int)ny - 1) return std::printf("%g %g of %u: %d %d\n", f0, f1, ny, lo, hi), 1;
                int seen = 0, passes = 0;                    // the walk of a pass of 32 lanes at a time, as in the kernels
                for (int r0 = lo;; r0 += pic::ROW_PASS) {
                    if (++passes > 32) return std::printf("%g %g of %u: the walk does not end\n", f0, f1, ny), 1;
                    for (int lane = 0; lane < 32; ++lane) seen += r0 + lane <= hi;
                    if (!pic::rows_after(r0, hi)) break;
                }
                int want = 0;
                for (int r = 0; r < (int)ny; ++r) want += !((float)r < f0) && !((float)r > f1);
                if (seen != want) return std::printf("%g %g of %u: %d rows, not %d\n", f0, f1, ny, seen, want), 1;
            }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_rows_are_cut_to_the_grid_without_overflow(tmp_path):
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-fsanitize=undefined,float-cast-overflow", "-fno-sanitize-recover=all", "-I",
                    os.path.join(ROOT, "paper_2607_26005_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
