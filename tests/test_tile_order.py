"""The rule by which a call's tiles are drawn with the horizon first, on the host: only where that is another order than row by row and
the launch is small."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
SOURCE = r"""
#include <cstdio>
#include "pic_types.h"
int main() {
    const int sm = 148, most = pic::HORIZON_FIRST_TILES * sm;
    const struct { int H, W, tiles; bool want; } cases[] = {
        {64, 64, 1000, false}, {17, 33, 1000, false}, {64, 128, 1000, false}, {40, 192, 1000, false},     // one row of tiles alike
        {54, 96, 1000, true}, {64, 68, 1000, true}, {16, 1000, 1000, true},                              // a narrower last column
        {65, 64, 1000, true}, {128, 128, 1000, true}, {216, 384, 1000, true},                            // several rows
        {54, 96, most, true}, {54, 96, most + 1, false}, {128, 128, most, true}, {128, 128, most + 1, false}};
    for (auto& c : cases)
        if (pic::draws_horizon_first(c.H, c.W, c.tiles, sm) != c.want) return std::printf("%d x %d, %d tiles\n", c.H, c.W, c.tiles), 1;
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "vector_types.h")), reason="needs g++ and the CUDA headers")
def test_horizon_first_only_where_it_is_another_order(tmp_path):
    src, exe = tmp_path / "order.cpp", tmp_path / "order"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-I", CUDA, "-I", os.path.join(ROOT, "paper_2607_26005_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
