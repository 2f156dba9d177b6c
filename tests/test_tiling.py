"""The tiling of a frame (32-pixel columns, 16- and 8-pixel strips) on the CPU:
csrc/pc_internal.h's own functions, compiled into a small program.  Every pixel
of every band belongs to exactly one tile, no tile starts outside, there are
never more tiles than 32-pixel columns make, the staged rows of a warp fall
into different shared-memory banks, and the planes fit the size requested.  A
band of a frame stages every row its windows read and none after them, which
the host entry may still be copying in."""
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
// Bands of tile rows of an H x W frame, as the host entry cuts them; the ranges up
// to `halo` rows past a band are on the device when its tiles run.
static int check_bands(int H, int W, int th, int halo, int bands) {
    const int rows_t = (H + th - 1) / th;
    for (int b = 0; b < bands; b++) {
        const int row0 = rows_t * b / bands * th, end = rows_t * (b + 1) / bands * th, row1 = end < H ? end : H;
        const int copied = row1 + halo < H ? row1 + halo : H;
        const Tiling t = tiling_of(row1 - row0, W, th, true);
        for (int i = 0; i < t.full + t.n16 + t.n8; i++) {
            const TilePos p = tile_pos(t, i, th);
            const int first = row0 + p.vb, last = first + ((32 * th) >> p.lg) - 1;  // the tile's rows, its overhang too
            const int limit = staged_end(row1, halo, H);
            const int staged = last + halo < limit ? last + halo : limit - 1;       // last row it reads
            const int live = last < row1 ? last : row1 - 1;                         // last row it computes
            if (staged >= copied) return 1;
            if (staged < (live + halo < H ? live + halo : H - 1)) return 2;
        }
    }
    return 0;
}
int main() {
    const int frames[][2] = {{1000, 480}, {1270, 720}, {1912, 1080}, {517, 1003}, {645, 481}, {657, 333}, {640, 480}, {9, 77}};
    for (auto [W, H] : frames)
        for (int th : {8, 4})
            for (int halo : {1, 3, 7, 14, 24})
                for (int bands = 1; bands <= 8; bands++)
                    if (int e = check_bands(H, W, th, halo, bands)) {
                        printf("%d x %d, th %d, halo %d, %d bands: %d\n", W, H, th, halo, bands, e);
                        return 1;
                    }
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
                if (fit_smem_bytes(c, th, tw < 32) < need) { printf("planes of %d, halo %d\n", tw, halo); return 1; }
                // without strips no more than the 32-pixel tile, rounded up to 8 bytes
                if (tw == 32 && fit_smem_bytes(c, th, false) >= need + 8) { printf("halo %d: too much\n", halo); return 1; }
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
