"""Blocks at the sizes where the tiles, splits and dispatch rules of the kernels end: one row or column
more than a tile holds, widths that leave padded operand planes, reductions of one row and of many.
Everything is compared with the float64 oracle under the stated tolerances (tests/parity.py: 1e-4 in the
strict mode, 2e-2 outputs and 5e-2 gradients in the bf16 mode), which bound rounding at any size here:
the longest sum has 1224 products."""
from dataclasses import replace

import pytest

from paper_1707_04585_b200 import binding as B
from paper_1707_04585_b200 import synthetic as syn
from tests import helpers as hp
from tests import test_gpu_parity as tp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = B.Context(0)
    yield c
    B.revnet_check_device(c)
    c.close()


@pytest.mark.parametrize("kind,N,H,W,c,w", [
    ("basic", 2, 3, 3, 8, 0),             # one operand plane, less than one tile
    ("basic", 2, 281, 283, 8, 0),         # rows longer than a tile; nine tiles per CTA, one operand segment
    ("basic", 3, 2, 200, 24, 0),          # three planes, two-row images
    ("basic", 6, 9, 11, 40, 0),           # five planes
    ("basic", 4, 13, 13, 56, 0),          # seven planes, 56 of 64 output columns
    ("basic", 2, 16, 16, 64, 0),          # the widest layer with its BN and ReLU inside
    ("basic", 1, 103, 103, 88, 0),        # column reductions in two levels: 121 records, the last group one CTA
    ("bottleneck", 6, 9, 9, 32, 12),      # 1x1; rows of 48 bytes: 16-byte accesses
    ("bottleneck", 10, 23, 9, 128, 32),   # one column group: four warp groups on alternate tiles, records left to the consumer
    ("bottleneck", 10, 23, 9, 128, 64),   # two column groups
    ("bottleneck", 10, 23, 9, 160, 96),   # three
    ("bottleneck", 1, 9, 11, 128, 8),     # BN inside the wide 1x1: less than one tile, one 16-column group
    ("bottleneck", 3, 61, 107, 448, 128), # 153 tiles: some CTAs take two; seven chunks through three raw slots, four column groups
    ("bottleneck", 1, 97, 99, 520, 8),    # streaming kernels with 32-byte accesses: 65 octets of channels, three rows per pass
    ("bottleneck", 8, 9, 9, 136, 72),     # weight packs with padded rows (136 -> 256, 72 -> 80) and columns (136 -> 144)
])
def test_bf16_blocks_at_tile_edges(ctx, kind, N, H, W, c, w):
    tp.run_block_case(ctx, syn.BlockCfg(N, H, W, c, w, kind, seed=900 + c), 0, jitter=True, inplace=True)


@pytest.mark.parametrize("kind,N,H,W,c,w", [
    ("basic", 1, 5, 13, 4, 0),            # direct 3x3: one tile, half of it inside the image, outputs 4 of 16; 65 pixels in the weight gradient
    ("basic", 1, 275, 275, 16, 0),        # direct 3x3: 16-row tiles, the last one of 3 rows
    ("basic", 1, 150, 253, 20, 0),        # direct 3x3: 20 of 32 outputs; weight gradient by the GEMM, in 32-column tiles (rows too long for strips)
    ("basic", 1, 139, 137, 36, 0),        # direct 3x3: two groups of outputs, the second of 4; weight gradient of the first layer by the GEMM, in 64-column tiles
    ("basic", 2, 11, 7, 68, 0),           # two column tiles, the second of 4 columns
    ("basic", 16, 5, 4, 8, 0),            # direct 3x3: eight images per tile, one column of warps
    ("basic", 5, 7, 6, 20, 0),            # two images per tile, the last one of a tile missing
    ("basic", 75, 24, 16, 16, 0),         # direct 3x3, eight warps in two row groups: the second one of the last tile lies below the image
    ("basic", 9, 20, 7, 8, 0),            # the same with narrow images and four warps
    ("basic", 1, 33, 17, 100, 0),         # four chunks of input channels (the last of 4), four groups of outputs
    ("basic", 1, 119, 122, 132, 0),       # column reductions in two levels, two slabs: 121 records (statistics) and 242 (backward sums)
    ("bottleneck", 1, 277, 275, 16, 4),   # 1x1 GEMMs onto 4 and 16 channels in 256-row tiles, the last one of 143
    ("bottleneck", 1, 277, 275, 32, 20),  # ... onto 20 and 32
    ("bottleneck", 1, 195, 196, 64, 36),  # ... onto 36 and 64 in 128-row tiles, the last one of 76
    ("bottleneck", 1, 3, 3, 132, 4),      # column sums of nine rows: two slabs of 17 and 16 quads, and one quad
    ("bottleneck", 1, 97, 99, 520, 8),    # 32-byte accesses in the streaming kernels
    ("bottleneck", 2, 37, 41, 260, 136),  # three slabs (22, 22, 21), several row ranges; sums of 1224 products
])
def test_strict_blocks_at_tile_edges(ctx, kind, N, H, W, c, w):
    tp.run_block_case(ctx, syn.BlockCfg(N, H, W, c, w, kind, seed=900 + c), 1, jitter=True, inplace=True)


@pytest.mark.parametrize("img,k,stem_c", [
    (10, 3, 40),       # 3x3 row kernel: rows of ten pixels in turns of twelve, a second channel group of 8 lanes
    (48, 7, 72),       # 7x7: rows of 24 pixels in turns of seven, three channel groups of the weight gradient
    (56, 7, 8),        # one channel per lane, rows of 28 pixels in segments of eight
])
def test_stems_at_tile_edges(ctx, img, k, stem_c):
    cfg = replace(hp.tiny_stack("bottleneck", k == 7, N=3), img=img, stem_cout=stem_c)
    tp.run_stack_case(ctx, cfg, 1)
    tp.ORACLE_RUNS.clear()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("N,H,cin,cout,stride,split", [
    (3, 6, 8, 24, 2, False),              # 27 pixels in each parity class of the data gradient
    (2, 10, 40, 72, 2, False),
    (2, 9, 24, 136, 1, False),
    (5, 14, 48, 80, 2, True),             # halves of 24 and 40: the staged epilogue in both directions
    (3, 10, 24, 400, 1, True),            # halves of 12 and 200, four column tiles
    (4, 20, 96, 224, 2, True),            # halves of 48 and 112: 16-column groups on a pair, with and without a partner tile
])
def test_transitions_at_tile_edges(ctx, mode, N, H, cin, cout, stride, split):
    tp.run_transition_case(ctx, mode, N, H, cin, cout, 3, stride, split)
