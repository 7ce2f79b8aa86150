"""Tiles of the strict-mode 3x3 kernel, on the host: the geometry that the kernel runs with (csrc/conv_direct.cuh, compiled here
by itself) is walked lane by lane.  Every row that a lane stores, and so every row of the coupling partner that it
reads, must lie inside the tensor, and every output must be stored exactly once."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1707_04585_b200", "csrc")

PROGRAM = r"""
#include "conv_direct.cuh"
#include <stdio.h>
#include <stdlib.h>

static long shapes, below;      // shapes the kernel takes; warps whose first row lies below the image

static void walk(int N, int H, int W, int Ci, int Co) {
    DirectGeom g;
    if (!direct_shape(N, H, W, Ci, Co, 148, g)) return;
    shapes++;
    const int smem = (9 * g.kc * g.CB * 16 + 2 * (g.gx * 4 + 2) * (g.gy * 8 + 2) * g.gi * g.pitch) * 4;
    const int wpx = g.NW / g.CB, nb = g.CB * 16, nbs = (Co + nb - 1) / nb;
    if (smem > 160 * 1024 || wpx != g.gx * g.gy * g.gi || g.tiles != g.tx * g.ty * ((N + g.gi - 1) / g.gi)) { printf("bad geometry %d %d %d %d %d\n", N, H, W, Ci, Co); exit(1); }
    const size_t P = (size_t)N * H * W;
    std::vector<unsigned char> stored(P * Co, 0);
    for (int by = 0; by < nbs; by++)
        for (int t = 0; t < g.tiles; t++) {
            const int x0 = t % g.tx * g.gx * 4, y0 = t / g.tx % g.ty * g.gy * 8, i0 = t / (g.tx * g.ty) * g.gi;
            for (int warp = 0; warp < g.NW; warp++) {
                const int wt = warp % wpx, wc = warp / wpx, wx = wt % g.gx, wy = (wt / g.gx) % g.gy, wi = wt / (g.gx * g.gy);
                if (y0 + wy * 8 >= H) below++;
                for (int lane = 0; lane < 32; lane++) {
                    const int n = by * nb + wc * 16 + 2 * (lane >> 2), x = x0 + wx * 4 + (lane & 3), y = y0 + wy * 8, i = i0 + wi;
                    const int live = direct_live_rows(g, n, x, y, i);
                    if (live <= 0) continue;
                    const size_t row = ((size_t)i * H + y) * W + x;
                    for (int r = 0; r < 8; r++) {
                        const size_t at = row + (size_t)(r < live ? r : 0) * W;       // partner row; the stored row for r < live
                        if (at >= P || y + (r < live ? r : 0) >= H || n + 1 >= Co) { printf("N %d H %d W %d Co %d: image %d row %d column %d output %d reads row %zu of %zu\n", N, H, W, Co, i, y, x, n, at, P); exit(1); }
                        if (r < live) { stored[at * Co + n]++; stored[at * Co + n + 1]++; }
                    }
                }
            }
        }
    for (unsigned char c : stored) if (c != 1) { printf("N %d H %d W %d Co %d: an output is stored %d times\n", N, H, W, Co, (int)c); exit(1); }
}

int main() {
    const int Ns[] = {1, 3, 37, 80}, Ws[] = {1, 3, 4, 5, 7, 8, 9, 15, 16, 17, 20, 33}, Cs[] = {4, 16, 20, 68};
    for (int N : Ns) for (int W : Ws) for (int C : Cs) for (int H = 1; H <= 41; H++) walk(N, H, W, C, C);
    walk(75, 24, 16, 16, 16); walk(128, 24, 24, 16, 16); walk(1, 275, 275, 16, 16); walk(2, 150, 253, 8, 20);
    printf("%ld %ld\n", shapes, below);
    return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.exists("/usr/local/cuda/include/cuda_runtime.h"), reason="no g++ or CUDA headers")
def test_direct_kernel_rows_stay_inside_the_tensors(tmp_path):
    src, exe = tmp_path / "walk.cpp", tmp_path / "walk"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I/usr/local/cuda/include", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    shapes, below = map(int, out.stdout.split())
    assert shapes > 1000 and below > 1000          # the sweep holds the sizes in question
