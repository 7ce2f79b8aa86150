"""Launch geometry of the fused BN-ReLU-conv kernel, on the host: csrc/conv_fused_shape.cuh, compiled here by itself, as the
kernel's launcher uses it."""
import os
import shutil
import subprocess

import pytest

from tests import test_gpu_fused_rings as rings

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1707_04585_b200", "csrc")

PROGRAM = r"""
#include "conv_fused_shape.cuh"
#include <stdio.h>
#include <stdlib.h>

static int tiles_of(const FusedGeom &g) { return (g.chunk + 127) / 128; }

// A build thread fills its rows' entries of a segment's table once every warp has built the segment that had the same operand buffer before
// (nseg back).  Any other warp may then still be 1 .. nseg - 1 segments behind: if it reads the same table, the rows in question must be its own.
static bool tables_safe(const FusedShape &s) {
    const FusedGeom &g = s.g;
    if (g.k == 1 || tiles_of(g) <= g.S) return true;
    bool shared = false;                                  // a row whose threads sit in two warps
    for (int r = 0; r < g.RS; r++) shared = shared || r * g.nit / 32 != (r * g.nit + g.nit - 1) / 32;
    for (int d = 1; d < g.nseg; d++) if (shared && d % g.tabs == 0) return false;
    return true;
}

int main(int argc, char **) {
    if (argc > 1) {       // shapes from standard input
        int N, H, W, ci, co, k, mode;
        while (scanf("%d %d %d %d %d %d %d", &N, &H, &W, &ci, &co, &k, &mode) == 7) {
            FusedShape s;
            if (!fused_shape(Geom{N, H, W}, ci, co, k, 148, mode, true, s)) { printf("0 0 0\n"); continue; }
            printf("%d %d %d\n", tiles_of(s.g), s.g.S, mode == kInBwd ? (int)fused_folds(s) : s.g.nseg);
        }
        return 0;
    }
    long taken = 0, segmented = 0, two = 0;
    const int Ns[] = {1, 5, 37, 100, 128, 700}, Hs[] = {1, 7, 24, 48, 130, 400};
    for (int N : Ns) for (int H : Hs) for (int W = 1; W < 700; W += 1 + W / 6) for (int ci = 8; ci <= 64; ci += 8) for (int co : {4, 16, 24, 32, 64, 256})
        for (int k = 1; k <= 3; k += 2) for (int mode = 0; mode < 4; mode++) {
            FusedShape s;
            if (!fused_shape(Geom{N, H, W}, ci, co, k, 148, mode, true, s)) continue;
            const FusedGeom &g = s.g;
            taken++; segmented += tiles_of(g) > g.S; two += g.tabs == 2;
            if (!tables_safe(s)) { printf("N %d H %d W %d %d->%d k %d mode %d: two warps share a table that one may rewrite\n", N, H, W, ci, co, k, mode); return 1; }
            const int used = 1024 + k * k * g.wtile_bytes + s.EW * g.aux_slots * kAuxBytes + g.op_bytes + g.raw_slots * g.raw_bytes + g.tabs * g.tab_bytes + (int)sizeof(FusedShared);
            if (used > s.smem || s.smem > 227 * 1024) { printf("N %d H %d W %d %d->%d k %d mode %d: %d bytes used, %d asked for\n", N, H, W, ci, co, k, mode, used, s.smem); return 1; }
        }
    printf("%ld %ld %ld\n", taken, segmented, two);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists("/usr/local/cuda/include/cuda_runtime.h"):
        pytest.skip("no g++ or CUDA headers")
    d = tmp_path_factory.mktemp("shapes")
    (d / "shapes.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I/usr/local/cuda/include", "-I" + CSRC, str(d / "shapes.cpp"), "-o", str(d / "shapes")], check=True)
    return str(d / "shapes")


def test_tables_of_pixels_and_shared_memory(program):
    out = subprocess.run([program], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
    taken, segmented, two = map(int, out.stdout.split())
    assert taken > 50000 and segmented > 5000 and two > 1000          # the sweep holds the sizes in question


@pytest.mark.parametrize("kind,N,H,W,c,segments,buffers", rings.SEGMENTED)
def test_segmented_cases_have_the_segments_that_they_claim(program, kind, N, H, W, c, segments, buffers):
    shapes = "".join(f"{N} {H} {W} {c} {c} 3 {mode}\n" for mode in (1, 2))          # data gradient; forward on the fixed-point state
    out = subprocess.run([program, "-"], input=shapes, capture_output=True, text=True, check=True).stdout.split()
    for tiles, S, nseg in (map(int, out[i:i + 3]) for i in (0, 3)):
        assert nseg == buffers and -(-tiles // S) == segments


def test_fold_cases_fold_or_not_as_they_claim(program):
    shapes = "".join(f"{N} {H} {W} {c} {c} 3 3\n" for N, H, W, c, _ in rings.FOLDS)
    out = subprocess.run([program, "-"], input=shapes, capture_output=True, text=True, check=True).stdout.split()
    assert [int(v) for v in out[2::3]] == [int(folds) for *_, folds in rings.FOLDS]
