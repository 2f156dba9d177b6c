"""The tiling of a frame (32-pixel columns, 16- and 8-pixel strips) on the CPU:
csrc/pc_internal.h's own functions, compiled into a small program.  Every pixel
of every band belongs to exactly one tile, no tile starts outside, there are
never more tiles than 32-pixel columns make, the staged rows of a warp fall
into different shared-memory banks, and the planes fit the size requested."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdio>
#include <vector>
#include "pc_internal.h"
using namespace pcurv;
static int check(int rows, int W, int th, bool strips) {
    const Tiling t = tiling_of(rows, W, th, strips);
    const int n = t.full + t.n16 + t.n8;
    if (n > ((W + 31) / 32) * ((rows + th - 1) / th)) return 1;
    std::vector<unsigned char> hit((size_t)rows * W, 0);
    for (int i = 0; i < n; i++) {
        const TilePos p = tile_pos(t, i, th);
        if (p.lg < (strips ? 3 : 5) || p.lg > 5 || p.ub < 0 || p.vb < 0 || p.ub >= W || p.vb >= rows) return 2;
        const int tw = 1 << p.lg, h = (32 * th) >> p.lg;
        for (int y = p.vb; y < p.vb + h && y < rows; y++)
            for (int x = p.ub; x < p.ub + tw && x < W; x++)
                if (hit[(size_t)y * W + x]++) return 3;
    }
    for (unsigned char h : hit)
        if (h != 1) return 4;
    return 0;
}
int main() {
    for (int th : {8, 4, 2, 1})
        for (int strips = 0; strips <= (th >= 4); strips++)
            for (int W = 1; W <= 130; W++)
                for (int rows : {1, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 47, 64, 65, 241})
                    if (int e = check(rows, W, th, strips)) { printf("rows %d W %d th %d strips %d: %d\n", rows, W, th, strips, e); return 1; }
    for (int halo = 1; halo <= 24; halo++) {
        FitConfig c{};
        c.r = halo;
        c.rn = 1;
        for (int tw : {32, 16, 8}) {
            const int pitch = tile_pitch(tw, halo);
            unsigned banks = 0;
            for (int l = 0; l < 32; l++) banks |= 1u << ((l / tw * pitch + l % tw) % 32);
            if (pitch < tw + 2 * halo || banks != 0xffffffffu) { printf("pitch %d of %d, halo %d\n", pitch, tw, halo); return 1; }
            for (int th : {8, 4}) {
                const size_t rows = 32 * th / tw + 2 * halo, need = pitch * rows * 8 + rows * tw * 4;
                if (fit_smem_bytes(c, th, true) < need) { printf("planes of %d, halo %d\n", tw, halo); return 1; }
            }
        }
    }
    printf("ok\n");
    return 0;
}
"""


def test_every_pixel_belongs_to_one_tile(tmp_path):
    include = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "tiling.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "tiling"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I" + include,
                    "-I" + os.path.join(ROOT, "paper_1707_00385_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
