"""Geometry of the strict mode's weight gradients in strips of image rows, on the host: csrc/conv_strips.cuh, compiled here by itself."""
import os
import shutil
import subprocess

import pytest

from tests import test_gpu_fused_rings as rings

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1707_04585_b200", "csrc")

PROGRAM = r"""
#include "conv_strips.cuh"
#include <stdio.h>
#include <stdlib.h>

static bool shape(int N, int H, int W, int Ci, int Co, WgStrip &p, int &ctas, int &threads, int &smem) {
    // (what the caller allocates behind the partials: the data gradient)
    const int most = (int)((size_t)N * H * W / (9 * Co));
    return wg_strip_shape(N, H, W, Ci, Co, 148, most > 1 ? most : 1, p, ctas, threads, smem);
}

int main(int argc, char **) {
    WgStrip p;
    int ctas, threads, smem;
    if (argc > 1) {       // shapes from standard input
        int N, H, W, ci, co;
        while (scanf("%d %d %d %d %d", &N, &H, &W, &ci, &co) == 5) printf("%d\n", shape(N, H, W, ci, co, p, ctas, threads, smem) ? 1 : 0);
        return 0;
    }
    long taken = 0;
    const int Ns[] = {1, 9, 40, 128, 700}, Cs[] = {4, 12, 16, 24, 36, 44, 48, 64};
    for (int N : Ns) for (int H = 1; H <= 60; H += 1 + H / 6) for (int W = 1; W <= 512; W += 1 + W / 5) for (int ci : Cs) for (int co : Cs) {
        if (!shape(N, H, W, ci, co, p, ctas, threads, smem)) continue;
        taken++;
        const size_t stage = (size_t)p.a_floats + p.g_floats, red = (size_t)p.R * p.sl * 9 * ci * co;
        const bool bad = threads != 96 * p.nb * p.R || threads > kWgStripThreads || smem > 200 * 1024 || (size_t)smem < 2 * stage * 4 || (p.R * p.sl > 1 && (size_t)smem < red * 4) ||
                         p.sl * p.pairs > 32 * (p.sl > 1 ? 1 : p.nb) || p.nb * 32 < p.pairs || p.R * p.sl > H;
        std::vector<int> seen((size_t)N * H, 0);
        for (int c = 0; c < ctas; c++)
            for (int s = c * p.per_cta; s < p.strips && s < (c + 1) * p.per_cta; s++) {
                const int n = s / p.per_img, y0 = s % p.per_img * p.BH, rows = H - y0 < p.BH ? H - y0 : p.BH;
                if ((rows + 2) * (W + 2) * ci > p.a_floats || rows * W * co > p.g_floats) { printf("N %d H %d W %d %d->%d: a strip does not fit its buffer\n", N, H, W, ci, co); return 1; }
                for (int sl = 0; sl < p.R * p.sl; sl++) for (int r = sl; r < rows; r += p.R * p.sl) seen[(size_t)n * H + y0 + r]++;
            }
        for (int v : seen) if (bad || v != 1) { printf("N %d H %d W %d %d->%d: bad geometry, or a row added %d times\n", N, H, W, ci, co, v); return 1; }
    }
    printf("%ld\n", taken);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists("/usr/local/cuda/include/cuda_runtime.h"):
        pytest.skip("no g++ or CUDA headers")
    d = tmp_path_factory.mktemp("strips")
    (d / "strips.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I/usr/local/cuda/include", "-I" + CSRC, str(d / "strips.cpp"), "-o", str(d / "strips")], check=True)
    return str(d / "strips")


def test_every_row_is_added_once_from_inside_its_buffer(program):
    out = subprocess.run([program], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    assert int(out.stdout) > 2000          # the sweep holds the sizes in question


def test_strip_cases_take_the_path_that_they_claim(program):
    shapes = "".join(f"{N} {H} {W} {c} {c}\n" for _, N, H, W, c, _ in rings.STRIPS)
    out = subprocess.run([program, "-"], input=shapes, capture_output=True, text=True, check=True).stdout.split()
    assert [int(v) for v in out] == [int(taken) for *_, taken in rings.STRIPS]
