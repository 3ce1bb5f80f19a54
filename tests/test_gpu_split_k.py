"""Small problems (fewer tiles than SMs) through both kernels that serve them: clusters sharing a tile's k-blocks
(B2C_SPLIT_K=1, the default) and the persistent kernel (0), against the oracle at the per-tensor budget."""
import numpy as np
import pytest
import torch

import oracle
from paper_2503_23186_b200 import workloads as wl
from parity import assert_close, dev_bf16, dev_f32, host

pytestmark = pytest.mark.gpu

# an odd number of tiles on pairs, one tile split eight ways, slices of 8 / 20 x 8 columns, 16- and 32-channel k-blocks, output parities
# with and without taps, more splits than a ragged share of k-blocks, several images per tile with a ragged last one,
# partial tiles too large to have an area beside the ring, two tiles per SM
SHAPES = [(50, 4, 4, 512, 512, 3, 1), (8, 4, 4, 256, 64, 3, 1), (3, 8, 8, 32, 32, 3, 1), (8, 32, 32, 16, 16, 3, 1), (2, 16, 16, 160, 160, 3, 1),
          (8, 8, 8, 128, 256, 3, 2), (8, 8, 8, 128, 256, 1, 2), (5, 16, 16, 32, 64, 3, 2), (6, 8, 8, 48, 96, 3, 1), (16, 8, 8, 2048, 512, 1, 1), (7, 4, 4, 640, 320, 3, 1), (33, 8, 8, 512, 256, 3, 1),
          (81, 32, 32, 16, 32, 3, 2), (75, 16, 16, 64, 64, 1, 1)]
# Layers whose plans split a tile, with what the plan has to be (forward, data gradient; None: whatever it is): parities through the
# exchange, in an area of its own and through the ring's memory, parities without taps, slices of 40, 24 and 8 columns, k-blocks of 32 and
# 16 channels, split pairs
SPLIT = [((50, 8, 8, 256, 512, 3, 2), dict(splits=2), dict(splits=2, overlap=1)), ((8, 8, 8, 256, 512, 3, 2), dict(splits=8), dict(splits=4, overlap=0)),
         ((8, 8, 8, 1024, 2048, 1, 2), dict(splits=4), dict(splits=2)), ((32, 8, 8, 160, 160, 3, 1), dict(splits=2, tile_channels=80, k_block=32), None),
         ((8, 8, 8, 512, 80, 3, 1), dict(splits=2, tile_channels=80), dict(splits=4, k_block=16)), ((24, 4, 4, 240, 512, 1, 2), None, dict(splits=2, tile_channels=48)),
         ((1, 4, 4, 128, 544, 1, 2), None, dict(splits=4, tile_channels=32, k_block=32)), ((39, 4, 4, 640, 480, 3, 1), dict(splits=4, tile_channels=96, pair=1), None),
         ((35, 4, 4, 224, 304, 3, 2), None, dict(splits=4, overlap=1, k_block=16))]
# B2C_SPLIT_K=0 on pairs: two threads that share units, and alternate units
PERSISTENT_PAIRS = [((8, 16, 16, 256, 256, 3, 1), dict(kind="shared-units", pair=1)), ((80, 16, 16, 128, 128, 3, 1), dict(kind="general", pair=1))]


@pytest.fixture(scope="module", params=["0", "1"], ids=["persistent", "split-k"])
def ctx(request):
    import os
    from paper_2503_23186_b200 import binding
    before = os.environ.get("B2C_SPLIT_K")
    os.environ["B2C_SPLIT_K"] = request.param
    try:
        c = binding.Context(0)
    finally:
        if before is None:
            del os.environ["B2C_SPLIT_K"]
        else:
            os.environ["B2C_SPLIT_K"] = before
    c.split_k = request.param == "1"
    yield c
    assert c.device_status() == 0
    c.close()


def _desc(N, H, W, C, K, R, st):
    from paper_2503_23186_b200 import binding
    return binding.conv_desc(N, H, W, C, K, R, st)


def _check_plan(ctx, shape, which, want):
    plan = ctx.conv2d_plan(_desc(*shape), which)
    assert want is None or all(plan[k] == v for k, v in want.items()), (shape, which, plan)


@pytest.mark.parametrize("shape", SHAPES + [s for s, _, _ in SPLIT] + [s for s, _ in PERSISTENT_PAIRS], ids=lambda s: "n{}h{}w{}c{}k{}r{}s{}".format(*s))
def test_forward_statistics_and_data_gradient(ctx, shape):
    N, H, W, C, K, R, st = shape
    if ctx.split_k:
        for s, fwd, dgrad in SPLIT:
            if s == shape:
                _check_plan(ctx, shape, "fwd", fwd)
                _check_plan(ctx, shape, "dgrad", dgrad)
    else:
        for s, want in PERSISTENT_PAIRS:
            if s == shape:
                _check_plan(ctx, shape, "fwd", want)
        assert ctx.conv2d_plan(_desc(*shape), "fwd")["kind"] != "one-wave"
    x, w, g = wl.conv_problem(40, *shape)
    pad, P = (R - 1) // 2, H // st
    y = torch.full((N, P, P, K), float("nan"), dtype=torch.bfloat16, device="cuda")
    stats = torch.zeros(2 * K, dtype=torch.float64, device="cuda")
    ctx.conv2d_fwd(_desc(*shape), dev_bf16(x), dev_bf16(w), y, ch_stats=stats)
    wd = torch.empty(w.size, dtype=torch.bfloat16, device="cuda")
    ctx.weight_pack_dgrad([(0, K, R * R, C)], dev_bf16(w).reshape(-1), wd)
    dx = torch.full(x.shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    ctx.conv2d_dgrad(_desc(*shape), dev_bf16(g), wd, dx)
    assert ctx.device_status() == 0
    assert_close(y, oracle.conv2d_fwd(x, w, st, pad), "y")
    assert_close(dx, oracle.conv2d_dgrad(g, w, x.shape, st, pad), "dx")
    ys = host(y).reshape(-1, K)   # sums of the stored values: fp32 over a tile's rows, fp64 across tiles
    np.testing.assert_allclose(host(stats)[:K], ys.sum(0), rtol=1e-5, atol=1e-3 * np.sqrt(ys.shape[0]))
    np.testing.assert_allclose(host(stats)[K:], (ys * ys).sum(0), rtol=1e-5)


@pytest.mark.parametrize("shape", [(250, 16, 16, 128, 256, 3, 2), (50, 4, 4, 512, 512, 3, 1), (64, 8, 8, 64, 160, 1, 1)], ids=lambda s: "n{}h{}w{}c{}k{}r{}s{}".format(*s))
def test_statistics_are_summed_in_fp32(ctx, shape):
    """Sums of squares of 32 rows in fp32, fp64 beyond: five levels of rounding to nearest leave a column about 1e-8 off in either
    direction.  Truncating additions, or chains of them (a square of a bf16 value ends in the same bits), lose 5e-8 and more."""
    N, H, W, C, K, R, st = shape
    x, w, _ = wl.conv_problem(43, *shape)
    P = H // st
    y = torch.empty((N, P, P, K), dtype=torch.bfloat16, device="cuda")
    stats = torch.zeros(2 * K, dtype=torch.float64, device="cuda")
    ctx.conv2d_fwd(_desc(*shape), dev_bf16(x), dev_bf16(w), y, ch_stats=stats)
    ys = y.double().reshape(-1, K)
    err = (stats[K:] / (ys * ys).sum(0) - 1).cpu().numpy()
    assert np.mean(np.abs(err)) <= 2.5e-8 and abs(np.mean(err)) <= 2e-8, (np.mean(np.abs(err)), np.mean(err))
    err = ((stats[:K] - ys.sum(0)) / ys.abs().sum(0)).cpu().numpy()
    assert np.mean(np.abs(err)) <= 1e-8, np.mean(np.abs(err))


def test_classifier_with_bias(ctx):
    shape = (70, 1, 1, 512, 128, 1, 1)
    x, w, _ = wl.conv_problem(41, *shape)
    bias = wl.rng_for(41, "bias").standard_normal(128).astype(np.float32)
    y = torch.full((70, 1, 1, 128), float("nan"), dtype=torch.float32, device="cuda")
    ctx.conv2d_fwd(_desc(*shape), dev_bf16(x), dev_bf16(w), y, bias=dev_f32(bias))
    assert ctx.device_status() == 0
    assert_close(y, oracle.conv2d_fwd(x, w, 1, 0) + bias, "logits", 1e-5, 1e-5)   # fp32 output: accumulation error only


@pytest.mark.parametrize("shape", [(50, 4, 4, 512, 512, 3, 1), (8, 8, 8, 128, 256, 3, 2), (8, 32, 32, 64, 64, 3, 1)], ids=lambda s: "n{}h{}w{}c{}k{}r{}s{}".format(*s))
def test_winds_down_on_timeout(ctx, shape):
    """A poll budget of one: the status word reports it, every CTA of the cluster leaves, the next launch is correct."""
    N, H, W, C, K, R, st = shape
    x, w, _ = wl.conv_problem(42, *shape)
    y = torch.zeros((N, H // st, W // st, K), dtype=torch.bfloat16, device="cuda")
    X, Wt = dev_bf16(x), dev_bf16(w)
    ctx.set_spin_limit(1)
    try:
        for _ in range(8):   # (a poll may suspend for longer than a short launch takes: one launch can get through without a time-out)
            ctx.conv2d_fwd(_desc(*shape), X, Wt, y)
        status = ctx.device_status()
    finally:
        ctx.set_spin_limit(1 << 22)
    assert status == 7   # B2C_ERR_DEVICE_TIMEOUT
    ctx.conv2d_fwd(_desc(*shape), X, Wt, y)
    assert ctx.device_status() == 0
    assert_close(y, oracle.conv2d_fwd(x, w, st, 1), "y after recovery")
