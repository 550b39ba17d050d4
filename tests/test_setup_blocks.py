"""The set-up kernel's division of its work, on the host: every entry of every camera's tables and frusta and every agent belongs to one
thread, and no thread has more than one, so that large images do not lengthen the chain of a call."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
SOURCE = r"""
#include <cstdio>
#include <vector>
#include "pic_types.h"
using namespace pic;
int main() {
    const int cams[] = {1, 3, 16}, sizes[][2] = {{1, 1}, {64, 64}, {64, 640}, {704, 64}, {1080, 1920}, {4096, 4096}, {16384, 16384}}, agents[] = {1, 128, 129, 1000};
    for (int K : cams)
        for (auto& hw : sizes)
            for (int n : agents)
                for (int wanted = 0; wanted < 2; ++wanted) {
                    const int tiles = ((hw[0] + TILE - 1) / TILE) * ((hw[1] + TILE - 1) / TILE), per = (tiles + 1) * FRUSTUM_ENTRIES;
                    const SetupGrid grid = setup_grid(K, fast_div((uint32_t)K), hw[0], hw[1], wanted ? tiles : 0, n);
                    const int rays = ray_stride(hw[0]) + ray_stride(hw[1]);
                    const int blocks = setup_blocks(grid);
                    std::vector<int> table((size_t)K * rays, 0), entry((size_t)K * per, 0), agent(n, 0);
                    if (sizeof(float) * 4 * entry.size() != frusta_bytes(K, hw[0], hw[1])) return std::printf("%d entries do not fill the table\n", (int)entry.size()), 1;
                    int idle = 0;
                    for (int b = 0; b < blocks; ++b)
                        for (int t = 0; t < SETUP_THREADS; ++t) {
                            const SetupItem it = setup_item(grid, b, t);
                            if (it.camera < 0 || it.camera >= K || it.index < 0) return std::printf("block %d thread %d: camera %d item %d\n", b, t, it.camera, it.index), 1;
                            if (it.role == SETUP_TABLES) { if (it.index < rays) ++table[(size_t)it.camera * rays + it.index]; else ++idle; }
                            else if (it.role == SETUP_FRUSTA) { if (it.index < per) ++entry[(size_t)it.camera * per + it.index]; else ++idle; }
                            else if (it.index < n) ++agent[it.index];
                        }
                    for (int c : table) if (c != 1) return std::printf("an entry of the tables is made %d times\n", c), 1;
                    for (int c : entry) if (c != wanted) return std::printf("%d tiles: an entry is made %d times\n", tiles, c), 1;
                    for (int c : agent) if (c != 1) return std::printf("an agent is set up %d times\n", c), 1;
                    if (idle >= 2 * K * SETUP_THREADS) return std::printf("%d tiles: %d threads without an entry\n", tiles, idle), 1;
                }
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "vector_types.h")), reason="needs g++ and the CUDA headers")
def test_every_item_of_the_set_up_belongs_to_one_thread(tmp_path):
    src, exe = tmp_path / "setup.cpp", tmp_path / "setup"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-I", CUDA, "-I", os.path.join(ROOT, "paper_2607_26005_b200", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


RAYS = r"""
#include <cstdio>
#include "pic_types.h"
int main() {
    size_t most = 0;
    for (int n = 1; n <= 2048; ++n) {
        for (int from = 0; from < n; from += 16)             // a tile or a piece of one
            if (from + pic::TILE > pic::ray_stride(n)) return std::printf("%d: entries %d to %d of %d\n", n, from, from + pic::TILE, pic::ray_stride(n)), 1;
        if (n <= 512 && pic::table_bytes(16, n, n) > most) most = pic::table_bytes(16, n, n);
    }
    return most > pic::table_bytes(16, 512, 512);            // what pic_render_static reserves holds every smaller image's tables
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "vector_types.h")), reason="needs g++ and the CUDA headers")
def test_what_a_tile_reads_of_the_ray_tables_is_there(tmp_path):
    src, exe = tmp_path / "rays.cpp", tmp_path / "rays"
    src.write_text(RAYS)
    subprocess.run(["g++", "-std=c++17", "-I", CUDA, "-I", os.path.join(ROOT, "paper_2607_26005_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
