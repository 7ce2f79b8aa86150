"""Rounding of the strict mode's weight gradients (stored 3x3 layers, fp32): no larger than that of sums taken in the order of the
implicit GEMM, which adds the pixels in runs of 256 that 8, 4 or 2 warps share (at most 16, at most 32, more output channels)."""
import numpy as np
import pytest
import torch

from paper_1707_04585_b200 import binding as B

pytestmark = pytest.mark.gpu
SMS = 148


def gemm_order(a, g, Ci, Co):
    """fp32 sums over the last axis of a * g (float64, exact products) in the implicit GEMM's order for Ci -> Co channels."""
    P = a.shape[-1]
    bn, wk = (16, 8) if Co <= 16 else ((32, 4) if Co <= 32 else (64, 2))
    tiles = -(-9 * Ci // 64) * -(-Co // bn)
    splits = max(1, min(-(-SMS * 4 // tiles), -(-P // 256)))
    kps = -(-(-(-P // splits)) // 16) * 16
    splits = -(-P // kps)
    prod = torch.nn.functional.pad(a * g, (0, splits * kps - P)).view(-1, splits, kps // 16, wk, 16 // wk)
    acc = torch.zeros(prod.shape[:2] + (wk,), dtype=torch.float64, device=a.device)
    total = torch.zeros_like(acc)

    def fp32(x):
        return x.float().double()
    for chunk in range(kps // 16):
        for k in range(16 // wk):
            acc = fp32(acc + prod[:, :, chunk, :, k])
        if chunk % 16 == 15:
            total, acc = fp32(total + acc), torch.zeros_like(acc)
    acc = fp32(acc + total)
    part = acc[..., 0]
    for w in range(1, wk):
        part = fp32(part + acc[..., w])
    groups = []
    for z in range(min(8, splits)):
        s = part[:, z]
        for i in range(z + 8, splits, 8):
            s = fp32(s + part[:, i])
        groups.append(s)
    out = groups[0]
    for s in groups[1:]:
        out = fp32(out + s)
    return out


@pytest.mark.parametrize("Ci,Co,N,H,W", [
    (16, 16, 128, 32, 32), (16, 16, 256, 32, 32), (32, 32, 128, 16, 16), (32, 32, 256, 16, 16), (40, 40, 128, 32, 32), (48, 48, 128, 32, 32), (48, 48, 256, 32, 32),
    (32, 32, 64, 56, 56),       # rows of two runs
    (16, 16, 64, 56, 56),       # one round of the row slices is more than half of the shared memory
    (8, 8, 40, 31, 70),         # three runs per row, the last of four pixels
    (16, 64, 64, 32, 32),       # unequal channels
])
def test_strict_weight_gradient_error(Ci, Co, N, H, W):
    ctx = B.Context(0)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(100 + Ci + N)

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda")
    desc = B.TransitionDesc(N, H, W, Ci, Co, 3, 1, 0, 1e-5, 1, 0)
    x, dout = normal(N, H, W, Ci), [normal(N, H, W, Co // 2) for _ in range(2)]
    wt, gamma, beta = normal(Co, 3, 3, Ci) / np.sqrt(9 * Ci), torch.ones(Ci, device="cuda"), torch.zeros(Ci, device="cuda")
    din, dW, dg, db = torch.empty_like(x), torch.empty_like(wt), torch.empty_like(gamma), torch.empty_like(beta)
    ws = torch.empty(max(B.revnet_transition_workspace_bytes(ctx, desc)), dtype=torch.uint8, device="cuda")
    B.revnet_transition_bwd(ctx, desc, x, None, *dout, wt, gamma, beta, din, None, dW, dg, db, ws)
    torch.cuda.synchronize()
    B.revnet_check_device(ctx)
    ctx.close()
    x64 = x.double()
    var, mean = torch.var_mean(x64, dim=(0, 1, 2), unbiased=False)
    a = torch.relu((x64 - mean) / torch.sqrt(var + 1e-5))
    ap = torch.nn.functional.pad(a, (0, 0, 1, 1, 1, 1))
    g = torch.cat(dout, dim=3).double()
    rng = np.random.default_rng(Ci)
    got, want, order = [], [], []
    for _ in range(24):          # outputs (co, kh, kw, all ci) of 24 random taps
        co, kh, kw = int(rng.integers(Co)), int(rng.integers(3)), int(rng.integers(3))
        at = ap[:, kh:kh + H, kw:kw + W, :].reshape(-1, Ci).t().contiguous()
        gc = g[..., co].reshape(1, -1)
        want.append((at * gc).sum(1)); got.append(dW[co, kh, kw].double())
        order.append(gemm_order(at.float().double(), gc, Ci, Co))
    got, want, order = (torch.cat(t) for t in (got, want, order))
    mine, gemm = (float((t - want).norm() / want.norm()) for t in (got, order))
    # On top of the sums, the kernel's activated input is BN in fp32: three roundings of up to 2^-24 each (0.6 * 2^-24 rms), independent
    # from pixel to pixel, so relative to the sum of random signs 3^0.5 * 0.6 * 2^-24 = 6.2e-8.  A share of 192 to 1152
    # outputs: the ratio of two rms errors is known to 1.5 / sqrt(2 * 192) = 8 %.
    assert mine <= 1.08 * np.hypot(gemm, 6.2e-8), (mine, gemm)
