"""Edges of the average pool (image rows and channel vectors shared by a block) and of convolution plans: units of one ring slot on
256-channel tiles, filter rows that do not fill a tile of the weight gradient."""
import numpy as np
import pytest
import torch

import oracle
from paper_2503_23186_b200 import workloads as wl
from parity import assert_close, dev_bf16, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2503_23186_b200 import binding
    c = binding.Context(0)
    yield c
    assert c.device_status() == 0
    c.close()


# rows of threads per vector: one (many images, few channels; one position), up to 32, up to 256; positions that the rows do not divide,
# vectors that do not fill a block or straddle images
@pytest.mark.parametrize("n,hw,c", [(1, 1, 8), (3, 7, 48), (5, 16, 512), (2, 64, 128), (3, 49, 2048), (2, 300, 264), (9000, 4, 16), (70000, 1, 8), (1, 4096, 24), (257, 9, 136)])
def test_avgpool(ctx, n, hw, c):
    a = wl.normal_bf16(60, f"pool{hw}x{c}", (n, hw, c))
    pooled = torch.full((n, c), float("nan"), dtype=torch.bfloat16, device="cuda")
    ctx.avgpool_fwd(n, hw, c, dev_bf16(a), pooled)
    assert ctx.device_status() == 0
    assert_close(pooled, oracle.round_bf16(a.astype(np.float64).mean(1)), "pooled")


# one k-block per unit on 256-channel tiles (two issuing threads, one slot per unit), several units per walker; 64 -> 256 3x3
@pytest.mark.parametrize("shape", [(96, 16, 16, 64, 256, 1, 1), (40, 16, 16, 64, 256, 3, 1)], ids=["one-slot-units", "wide-3x3"])
def test_wide_tiles_with_statistics(ctx, shape):
    from paper_2503_23186_b200 import binding
    N, H, W, C, K, R, st = shape
    x, w, _ = wl.conv_problem(61, *shape)
    ref = oracle.conv2d_fwd(x, w, st, (R - 1) // 2)
    for _ in range(3):
        y = torch.full((N, H, W, K), float("nan"), dtype=torch.bfloat16, device="cuda")
        stats = torch.zeros(2 * K, dtype=torch.float64, device="cuda")
        ctx.conv2d_fwd(binding.conv_desc(*shape), dev_bf16(x), dev_bf16(w), y, ch_stats=stats)
        assert ctx.device_status() == 0
        assert_close(y, ref, "y")
        ys = host(y).reshape(-1, K)   # sums of the stored values: fp32 within a walker, fp64 across
        np.testing.assert_allclose(host(stats)[:K], ys.sum(0), rtol=1e-5, atol=1e-3 * np.sqrt(ys.shape[0]))
        np.testing.assert_allclose(host(stats)[K:], (ys * ys).sum(0), rtol=1e-5)


# walkers of 28 wide and 55 narrow tiles: chains of single squares in fp32 would come out 9e-8 and 5e-8 low (a square of a bf16 value
# ends in the same bits); sums over 32 rows in fp32 are about 1.1e-8 off, whatever the length of the walk
@pytest.mark.parametrize("shape", [(256, 32, 32, 32, 512, 1, 1), (1024, 32, 32, 16, 64, 1, 1)], ids=["wide", "narrow"])
def test_statistics_of_long_walks(ctx, shape):
    from paper_2503_23186_b200 import binding
    N, H, W, C, K, R, st = shape
    gen = torch.Generator(device="cuda")
    gen.manual_seed(64)
    x = torch.randn((N, H, W, C), generator=gen, device="cuda").to(torch.bfloat16)
    w = (torch.randn((K, R, R, C), generator=gen, device="cuda") * (2.0 / C) ** 0.5).to(torch.bfloat16)
    y = torch.empty((N, H, W, K), dtype=torch.bfloat16, device="cuda")
    stats = torch.zeros(2 * K, dtype=torch.float64, device="cuda")
    ctx.conv2d_fwd(binding.conv_desc(*shape), x, w, y, ch_stats=stats)
    assert ctx.device_status() == 0
    ys = y.reshape(-1, K)
    squares = sum((part.double() ** 2).sum(0) for part in ys.split(1 << 16))
    err = (stats[K:] / squares - 1).cpu().numpy()
    assert np.mean(np.abs(err)) <= 2e-8, np.mean(np.abs(err))


# 75 / 80 tiles on 148 SMs: equal runs of (tile, pixel chunk) pairs, a CTA finishing one tile and beginning the next; partial tiles;
# up to 32 filter rows, as a whole bank, as the rest of one, and with many CTAs on the same rows; 1x1 tiles of up to 160 channels
@pytest.mark.parametrize("shape", [(32, 8, 8, 640, 640, 3, 1), (28, 8, 8, 1280, 2048, 1, 1), (31, 8, 8, 640, 624, 3, 1), (6, 8, 8, 48, 16, 3, 1), (4, 8, 8, 32, 144, 3, 1), (4, 8, 8, 16, 80, 1, 2), (7, 2, 2, 640, 16, 3, 1), (12, 4, 4, 128, 32, 3, 1),
                                   (40, 32, 32, 32, 32, 1, 1), (35, 4, 4, 256, 256, 1, 1), (9, 8, 8, 128, 144, 1, 1), (9, 8, 8, 176, 64, 1, 1)], ids=lambda s: "n{}h{}c{}k{}r{}s{}".format(*(s[i] for i in (0, 1, 3, 4, 5, 6))))
def test_weight_gradient_tiles(ctx, shape):
    from paper_2503_23186_b200 import binding
    N, H, W, C, K, R, st = shape
    x, _, g = wl.conv_problem(62, *shape)
    ref = oracle.conv2d_wgrad(g, x, R, R, st, (R - 1) // 2)
    dw = torch.full((K, R, R, C), float("nan"), dtype=torch.float32, device="cuda")
    ctx.conv2d_wgrad(binding.conv_desc(*shape), dev_bf16(g), dev_bf16(x), dw)
    assert_close(dw, ref, "dw")
    ctx.conv2d_wgrad(binding.conv_desc(*shape), dev_bf16(g), dev_bf16(x), dw, accumulate=True)
    assert ctx.device_status() == 0
    assert_close(dw, 2 * ref, "dw accumulated")


def test_weight_gradient_of_a_bank_beyond_2_to_the_31_elements(ctx):
    """Row offsets into dw need 64 bits: rows before, around and behind element 2^31 of a 65536 x 32832 filter bank."""
    from paper_2503_23186_b200 import binding
    shape = N, H, W, C, K, R, st = 2, 8, 8, 32832, 65536, 1, 1
    r = wl.rng_for(63, "big-bank")
    x, g = (torch.from_numpy(r.standard_normal((N, H, W, ch), dtype=np.float32)).to(torch.bfloat16) for ch in (C, K))
    dw = torch.full((K, C), float("nan"), dtype=torch.float32, device="cuda")
    ctx.conv2d_wgrad(binding.conv_desc(*shape), g.cuda(), x.cuda(), dw)
    assert ctx.device_status() == 0
    assert bool(torch.isfinite(dw.sum(1)).all())   # every row was written
    mid = (1 << 31) // C
    rows = np.r_[0:4, mid - 4:mid + 4, K - 4:K]
    want = g.double().numpy().reshape(-1, K)[:, rows].T @ x.double().numpy().reshape(-1, C)
    assert_close(dw[torch.from_numpy(rows).cuda()], want, "dw rows")


# rows of threads that fill a block, that do not (20, 3 and 256 channel vectors), that a warp adds up with shuffles first
@pytest.mark.parametrize("n,hw,c,bound", [(128, 8, 256, 1e-8), (64, 8, 160, 1e-8), (312, 8, 24, 1e-8), (2, 4, 2048, 1e-8), (40, 16, 64, 2e-8), (800, 32, 16, 2e-8)])
def test_batchnorm_sums_are_accurate(ctx, n, hw, c, bound):
    """Sums of squares in fp32 over eight rows, over a thread's steps and over the rows of a warp, in fp64 beyond.  A rounding leaves
    2^-26 of the partial sum on average; they add up along three levels per step, and five more where a warp's rows meet."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(65)
    shape = (n, hw, hw, c)
    y = (1.5 * torch.randn(shape, generator=gen, device="cuda") + 0.5).to(torch.bfloat16)
    a = torch.empty_like(y)
    stats = torch.full((2 * c,), float("nan"), dtype=torch.float64, device="cuda")
    mean, invstd = torch.empty(c, device="cuda"), torch.empty(c, device="cuda")
    ones, zeros = torch.ones(c, device="cuda"), torch.zeros(c, device="cuda")
    ctx.bn_relu_fwd(n, hw, hw, c, y, stats, False, ones, zeros, None, True, 1e-5, a, mean, invstd)
    assert ctx.device_status() == 0
    yd = y.double().reshape(-1, c)
    err = (stats[c:] / (yd * yd).sum(0) - 1).cpu().numpy()
    assert np.mean(np.abs(err)) <= bound, np.mean(np.abs(err))
    err = ((stats[:c] - yd.sum(0)) / yd.abs().sum(0)).cpu().numpy()
    assert np.mean(np.abs(err)) <= bound, np.mean(np.abs(err))


def test_staged_backward_of_the_widest_layers_with_two_gradients(ctx):
    """2048 channels, two upstream gradients: three tensors per ring stage, which the reduction's partial sums use once it is empty."""
    n, hw, c = 10, 8, 2048
    r = wl.rng_for(66, "bn-wide")
    y, da1, da2 = (wl.to_bf16_grid(r.standard_normal((n * hw * hw, c))) for _ in range(3))
    gamma = (1.0 + 0.1 * r.standard_normal(c)).astype(np.float32)
    mean, _, invstd = oracle.bn_stats(y, 1e-5)
    mean, invstd = oracle.round_f32(mean), oracle.round_f32(invstd)
    dy_ref, dres_ref, dg_ref, db_ref = oracle.bn_relu_bwd(da1, da2, y, y, gamma, mean, invstd, True, True)
    mask = torch.from_numpy(np.packbits((y > 0).reshape(-1, 8), axis=1, bitorder="little").reshape(-1)).cuda()
    dy, dres = (torch.full((n * hw * hw, c), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    dg, db = torch.zeros(c, device="cuda"), torch.zeros(c, device="cuda")
    ws = torch.empty(ctx.bn_relu_bwd_workspace_bytes(c), dtype=torch.uint8, device="cuda")
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v, dtype=np.float32)).cuda()
    ctx.bn_relu_bwd(n, hw, hw, c, dev_bf16(da1), dev_bf16(da2), dev_bf16(y), None, dev(gamma), dev(mean), dev(invstd), True, dy, dres, dg, db, False, ws, relu_mask=mask)
    assert ctx.device_status() == 0
    assert_close(dy, dy_ref, "dy")
    assert_close(dres, dres_ref, "dres")
    assert_close(dg, dg_ref, "dgamma", 1e-5, 1e-5)   # fp32 over a few rows, fp64 beyond
    assert_close(db, db_ref, "dbeta", 1e-5, 1e-5)
