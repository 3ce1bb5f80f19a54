"""The persistent convolution kernel's epilogue in blocks (tiles of 64, 128 and 256 channels): last tiles with images missing, several images
in a tile, output parities without taps, several channel tiles, pairs, and the BatchNorm sums of what was stored."""
import numpy as np
import pytest
import torch

import oracle
from paper_2503_23186_b200 import workloads as wl
from parity import assert_close, dev_bf16, host

pytestmark = pytest.mark.gpu

SHAPES = [
    (5, 4, 4, 64, 256, 1, 1), (37, 2, 2, 128, 128, 1, 1), (3, 8, 8, 256, 512, 1, 1), (9, 32, 32, 16, 64, 1, 1),   # 1x1: images end inside a tile
    (3, 16, 16, 64, 256, 1, 2), (7, 8, 8, 256, 128, 3, 2),                                                        # stride 2: parities of dx without taps
    (9, 8, 8, 64, 64, 3, 1), (3, 32, 32, 64, 64, 3, 1), (80, 32, 32, 64, 64, 3, 1), (151, 16, 16, 64, 64, 3, 1),  # vertical and merged taps
    (13, 16, 16, 128, 128, 3, 1), (450, 16, 16, 128, 128, 3, 1), (5, 8, 8, 128, 256, 3, 1), (66, 8, 8, 256, 256, 3, 1),   # pairs, full-halo stages
]
# kind and columns per block where they are not 64 (forward with sums, data gradient); (13, 16, 16, 128, 128) has no room for blocks
BLOCKS = {(9, 32, 32, 16, 64, 1, 1): ("general", 32, 0), (5, 4, 4, 64, 256, 1, 1): ("shared-units", 64, 32), (3, 16, 16, 64, 256, 1, 2): ("shared-units", 64, 32),
          (9, 8, 8, 64, 64, 3, 1): ("general", 32, 32), (3, 32, 32, 64, 64, 3, 1): ("general", 32, 32), (80, 32, 32, 64, 64, 3, 1): ("merged-taps", 32, 32),
          (151, 16, 16, 64, 64, 3, 1): ("merged-taps", 32, 32), (13, 16, 16, 128, 128, 3, 1): ("general", 0, 0), (450, 16, 16, 128, 128, 3, 1): ("full-halo", 16, 16),
          (66, 8, 8, 256, 256, 3, 1): ("shared-units", 64, 0)}


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "n{}h{}w{}c{}k{}r{}s{}".format(*s))
def test_blocks_of_the_epilogue(shape, monkeypatch):
    from paper_2503_23186_b200 import binding
    monkeypatch.setenv("B2C_SPLIT_K", "0")
    N, H, W, C, K, R, st = shape
    ctx = binding.Context(0)
    try:
        d, P = binding.conv_desc(*shape), H // st
        plan, back = ctx.conv2d_plan(d, "fwd", sums=True), ctx.conv2d_plan(d, "dgrad")
        kind, cols, cols_back = BLOCKS.get(shape, (plan["kind"], 64, 64))
        assert (plan["kind"], plan["block_cols"], back["block_cols"]) == (kind, cols, cols_back), (plan, back)
        if N > 160:   # the oracle takes a share of the images: as many as differ, repeated
            small = wl.conv_problem(51, 9, H, W, C, K, R, st)
            x, w, g = np.tile(small[0], (N // 9, 1, 1, 1)), small[1], np.tile(small[2], (N // 9, 1, 1, 1))
        else:
            x, w, g = small = wl.conv_problem(51, *shape)
        guard = 64   # rows behind the output that must stay as they are
        y = torch.full((N * P * P + guard, K), 7.0, dtype=torch.bfloat16, device="cuda")
        stats = torch.zeros(2 * K, dtype=torch.float64, device="cuda")
        ctx.conv2d_fwd(d, dev_bf16(x), dev_bf16(w), y, ch_stats=stats)
        plain = torch.full_like(y, 7.0)
        ctx.conv2d_fwd(d, dev_bf16(x), dev_bf16(w), plain)
        src = dev_bf16(w).reshape(-1)
        w_dgrad = torch.empty_like(src)
        ctx.weight_pack_dgrad([(0, K, R * R, C)], src, w_dgrad)
        dx = torch.full((N * H * W + guard, C), 7.0, dtype=torch.bfloat16, device="cuda")
        ctx.conv2d_dgrad(d, dev_bf16(g), w_dgrad, dx)
        assert ctx.device_status() == 0
        for t in (y, plain, dx):
            assert bool((t[-guard:] == 7.0).all())
        if ctx.conv2d_plan(d, "fwd")["kind"] != "shared-units":   # (two issuing threads there: the order of a tile's fp32 sums is open)
            assert bool((y == plain).all())
        assert_close(plain, host(y), "without sums")
        y, dx = y[:-guard].view(N, P, P, K), dx[:-guard].view(N, H, W, C)
        n = small[0].shape[0]
        for first in range(0, N, n):
            assert_close(y[first:first + n], oracle.conv2d_fwd(small[0], w, st, (R - 1) // 2) if first == 0 else host(y[:n]), "y")
            assert_close(dx[first:first + n], oracle.conv2d_dgrad(small[2], w, small[0].shape, st, (R - 1) // 2) if first == 0 else host(dx[:n]), "dx")
        f = y.double().reshape(-1, K)
        # between fp64 additions a value meets at most 13 fp32 ones: two or three among a unit's rows, eight units, three between lanes (by rows,
        # without blocks: five and five for the squares and sums of one unit)
        assert bool(((stats[:K] - f.sum(0)).abs() <= 13 * 2.0 ** -24 * f.abs().sum(0)).all())
        assert bool(((stats[K:] - (f * f).sum(0)).abs() <= 13 * 2.0 ** -24 * (f * f).sum(0)).all())
    finally:
        ctx.close()


# 221 and 110 units per CTA: 64-channel tiles, one MMA per tap and merged taps
@pytest.mark.parametrize("shape", [(4096, 32, 32, 16, 64, 1, 1), (2048, 32, 32, 64, 64, 3, 1)], ids=lambda s: "n{}h{}w{}c{}k{}r{}s{}".format(*s))
def test_sums_over_many_units(shape):
    """Ones, and a small value in every row that a lane meets last: a running fp32 sum over all units of a CTA loses the small values once
    it is large; sums of a few units, added up on their own, hold them."""
    from paper_2503_23186_b200 import binding
    N, H, W, C, K, R, st = shape
    ctx = binding.Context(0)
    try:
        d = binding.conv_desc(*shape)
        plan = ctx.conv2d_plan(d, "fwd", sums=True)
        assert plan["block_cols"] == 32, plan
        per_cta = N * H * W // 128 // plan["ctas"]
        assert per_cta >= 50, plan
        # a lane adds up rows l, l + 8, l + 16 and l + 24 of its warp's 32, of which the last is small: a quarter of the last bit of one running sum
        small = 2.0 ** (np.ceil(np.log2(3 * (per_cta + 1))) - 26)
        x = torch.zeros((N, H, W, C), dtype=torch.bfloat16, device="cuda")
        pixel = torch.arange(W, device="cuda")   # (rows of a warp: 32 pixels of one image row)
        x[..., 0] = torch.where(pixel >= 24, small, 1.0).to(torch.bfloat16)
        w = torch.zeros((K, R, R, C), dtype=torch.bfloat16, device="cuda")
        w[:, R // 2, R // 2, 0] = 1.0
        y = torch.empty((N, H, W, K), dtype=torch.bfloat16, device="cuda")
        stats = torch.zeros(2 * K, dtype=torch.float64, device="cuda")
        ctx.conv2d_fwd(d, x, w, y, ch_stats=stats)
        assert ctx.device_status() == 0
        assert bool((y == x[..., :1]).all())
        want = N * H * (24 + 8 * small)
        # a lane's sums of four units, and their sum, are exact; the last units' share and three additions between lanes round, warps meet in fp64
        assert bool(((stats[:K] - want).abs() <= 4 * 2.0 ** -24 * want).all()), ((stats[:K] - want) / want).abs().max().item()
    finally:
        ctx.close()
