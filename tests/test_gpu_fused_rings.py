"""Fused BN-ReLU-conv layers (and, in the strict mode, the weight gradient in strips of image rows) at the sizes where their rings of input pieces and partner rows, their operand segments and the
pass of a gradient through the BN backward of the layer behind begin and end.  Compared with the float64 oracle under the
stated tolerances (bf16 mode: 2e-2 outputs, 5e-2 gradients; strict mode: 1e-4), which bound rounding at these sizes."""
import numpy as np
import pytest

from paper_1707_04585_b200 import binding as B
from paper_1707_04585_b200 import runner as R
from paper_1707_04585_b200 import synthetic as syn
from tests import test_gpu_parity as tp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    B.revnet_check_device(c)
    c.close()


# Basic blocks whose inner data gradient takes its input through the BN backward of the layer behind, or does not (tests/test_fused_shapes_host.py)
FOLDS = [
    (37, 15, 21, 24, True),               # one tile per CTA
    (3, 5, 110, 16, True),                # the largest halo: six rows per build thread, and
    (3, 5, 111, 16, False),               # one size on
]


@pytest.mark.parametrize("kind,N,H,W,c,w", [
    ("basic", 1, 1, 1, 8, 0),             # one pixel; one piece
    ("basic", 3, 5, 110, 16, 0),          # (see FOLDS)
    ("basic", 3, 5, 111, 16, 0),
    ("basic", 37, 15, 21, 24, 0),
    ("basic", 150, 33, 31, 16, 0),        # nine tiles per CTA: the range as one segment, the partner ring goes round
    ("basic", 64, 32, 32, 64, 0),         # four tiles per CTA as one segment, two pieces of the input in flight
    ("basic", 3, 40, 150, 48, 0),         # long rows: a halo of 152 rows, six planes
    ("single", 9, 30, 33, 40, 0),         # one layer per function: sums of the only layer left to the last step
    ("bottleneck", 64, 32, 32, 128, 32),  # 1x1 onto 128 columns: many tiles per CTA in segments of two, both rings go round
])
def test_fused_layers_at_ring_edges(ctx, kind, N, H, W, c, w):
    tp.run_block_case(ctx, syn.BlockCfg(N, H, W, c, w, kind, seed=700 + c), 0, jitter=True, inplace=True)


# 3x3 layers whose CTAs take their range in several operand segments, in one buffer or two in turn (tests/test_fused_shapes_host.py holds the last
# two numbers, segments and buffers, against the launch geometry).  With 24, 40, 48 and 56 channels the threads of a row sit in two warps
SEGMENTED = [
    ("single", 2415, 31, 3, 24, 3, 2),
    ("basic", 935, 31, 3, 40, 3, 2),
    ("single", 935, 31, 3, 48, 3, 2),
    ("basic", 213, 31, 11, 56, 3, 2),
    ("single", 3, 133, 485, 24, 2, 1),
    ("basic", 3, 226, 119, 40, 2, 1),
    ("single", 2, 17, 691, 40, 4, 1),
    ("basic", 7, 114, 77, 56, 2, 1),
    ("single", 100, 24, 30, 64, 2, 1),
    ("single", 2, 9, 600, 64, 3, 1),      # rows so long that one piece of the input at a time is all that fits beside the operand
]


@pytest.mark.parametrize("kind,N,H,W,c,segments,buffers", SEGMENTED)
def test_segments_in_turn(ctx, kind, N, H, W, c, segments, buffers):
    tp.run_block_case(ctx, syn.BlockCfg(N, H, W, c, 0, kind, seed=750 + c), 0, jitter=True, inplace=True)


@pytest.mark.parametrize("N,H,W,c", [(3, 226, 119, 40), (935, 31, 3, 48)])
def test_segments_in_turn_give_the_same_bits_every_time(ctx, N, H, W, c):
    b = syn.BlockCfg(N, H, W, c, 0, "single", seed=790)
    r, inp = R.BlockRunner(ctx, b, 0), syn.make_block_inputs(b)
    r.load(inp["params"])
    first = None
    for _ in range(8):
        y1, y2 = r.forward(inp["x1"], inp["x2"])
        x1, x2, dx1, dx2, grads = r.backward(y1, y2, inp["dy1"], inp["dy2"])
        out = dict(grads, y1=y1, y2=y2, x1=x1, x2=x2, dx1=dx1, dx2=dx2)
        first = first or out
        assert all(np.array_equal(out[k], first[k]) for k in first)


# Strict weight gradients; the last value: in strips (held against the launch geometry by tests/test_strip_shapes_host.py), or by the implicit GEMM
STRIPS = [
    ("basic", 2, 9, 5, 12, False),        # a few pixels: the GEMM
    ("basic", 300, 9, 5, 12, True),       # nine pairs of quads: three row slices of a warp, five idle lanes; rows of 3 + 2 pixels
    ("basic", 700, 1, 7, 4, True),        # one row: one slice
    ("basic", 150, 17, 16, 16, True),     # strips of a whole image, the last round of slices one row
    ("single", 250, 26, 9, 44, True),     # 121 pairs in four blocks, the last of 25
    ("single", 20, 60, 61, 48, True),     # the most pairs that it takes: five blocks, 15 warps; rows of two runs of products
    ("single", 20, 60, 61, 52, False),    # one quad more: the implicit GEMM
    ("single", 40, 31, 70, 8, True),      # three runs per row, the last of four pixels
    ("single", 1, 275, 275, 16, False),   # rows too long for a warp's slices in two buffers
]


@pytest.mark.parametrize("kind,N,H,W,c,strips", STRIPS)
def test_strict_weight_gradient_strips(ctx, kind, N, H, W, c, strips):
    tp.run_block_case(ctx, syn.BlockCfg(N, H, W, c, 0, kind, seed=800 + c), 1, jitter=True, inplace=True)
