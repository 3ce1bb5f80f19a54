"""Which kernel a convolution layer gets: the rules of the planner at layers where a wrong estimate costs much."""
import random

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2503_23186_b200 import binding
    c = binding.Context(0)
    yield c
    c.close()


def _plan(ctx, which, shape):
    from paper_2503_23186_b200 import binding
    return ctx.conv2d_plan(binding.conv_desc(*shape), which)


# k-blocks of 16 or 32 channels whose taps share their loads: one tile per CTA, each tap loaded for itself, takes 1.2 to 1.7 times as long
@pytest.mark.parametrize("which,shape", [("dgrad", (25, 16, 16, 512, 784, 3, 1)), ("fwd", (17, 32, 32, 160, 160, 3, 1)), ("fwd", (6, 32, 32, 480, 512, 3, 1)),
                                         ("fwd", (5, 32, 32, 608, 320, 3, 1)), ("dgrad", (70, 16, 16, 256, 544, 3, 1))])
def test_narrow_k_blocks_stay_in_the_persistent_kernel(ctx, which, shape):
    assert _plan(ctx, which, shape)["kind"] != "one-wave"


@pytest.mark.parametrize("which,shape,splits", [("fwd", (50, 4, 4, 512, 512, 3, 1), 4), ("fwd", (313, 4, 4, 336, 64, 3, 1), 2), ("fwd", (382, 8, 8, 544, 48, 1, 1), 1)])
def test_few_tiles_go_to_the_one_wave_kernel(ctx, which, shape, splits):
    plan = _plan(ctx, which, shape)
    assert plan["kind"] == "one-wave" and plan["splits"] >= splits, plan


# Every kernel of the forward pass whose waits run out: the persistent ones (B2C_SPLIT_K=0) on pairs and single CTAs, with shared and alternate
# units, merged taps and full-halo stages, and the one-wave kernel with clusters and with two tiles per SM
@pytest.mark.parametrize("split_k,shape,want", [
    ("0", (16, 16, 16, 256, 256, 3, 1), dict(kind="shared-units", pair=1)), ("0", (100, 16, 16, 128, 128, 3, 1), dict(kind="general", pair=1)),
    ("0", (400, 16, 16, 128, 128, 3, 1), dict(kind="full-halo", pair=1)), ("0", (80, 32, 32, 64, 64, 3, 1), dict(kind="merged-taps")),
    ("0", (4, 16, 16, 128, 256, 3, 1), dict(kind="shared-units", pair=0)), ("0", (8, 32, 32, 64, 128, 3, 2), dict(kind="general", pair=0)),
    ("1", (8, 8, 8, 256, 512, 3, 2), dict(kind="one-wave", splits=8)), ("1", (75, 16, 16, 64, 64, 1, 1), dict(kind="one-wave", ctas=150)),
], ids=lambda v: v if isinstance(v, str) else "n{}h{}w{}c{}k{}r{}s{}".format(*v) if isinstance(v, tuple) else "-".join(map(str, v.values())))
def test_winds_down_on_timeout(split_k, shape, want, monkeypatch):
    """A poll budget of one: the status word reports it, every CTA leaves, and the next launch gives what one before gave."""
    from paper_2503_23186_b200 import binding
    monkeypatch.setenv("B2C_SPLIT_K", split_k)
    c = binding.Context(0)
    N, H, W, C, K, R, st = shape
    plan = _plan(c, "fwd", shape)
    assert all(plan[k] == v for k, v in want.items()), plan
    gen = torch.Generator(device="cuda")
    gen.manual_seed(70)
    x = torch.randn((N, H, W, C), generator=gen, device="cuda").to(torch.bfloat16)
    w = (torch.randn((K, R, R, C), generator=gen, device="cuda") * (2.0 / (R * R * C)) ** 0.5).to(torch.bfloat16)
    d = binding.conv_desc(*shape)
    good, y = (torch.full((N, H // st, W // st, K), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    c.conv2d_fwd(d, x, w, good)
    assert c.device_status() == 0
    c.set_spin_limit(1)
    try:
        for _ in range(8):
            c.conv2d_fwd(d, x, w, y)
        assert c.device_status() == 7   # B2C_ERR_DEVICE_TIMEOUT
    finally:
        c.set_spin_limit(1 << 22)
    y.fill_(float("nan"))
    c.conv2d_fwd(d, x, w, y)
    assert c.device_status() == 0
    diff = (y.float() - good.float()).norm() / good.float().norm()
    if want["kind"] == "shared-units":   # two threads issue into one accumulator: sums in either order, a few bf16 values one step (2^-8) apart
        assert diff.item() <= 1e-3, diff.item()
    else:
        assert diff.item() == 0.0, diff.item()
    c.close()


@pytest.mark.parametrize("shape", [(32, 8, 8, 640, 640, 3, 1), (28, 8, 8, 1280, 2048, 1, 1), (31, 8, 8, 640, 624, 3, 1)], ids=lambda s: "n{}h{}w{}c{}k{}r{}s{}".format(*s))
def test_weight_gradients_in_equal_runs(ctx, shape):
    """The layers with which the parity and wind-down tests mean the kernel that walks several tiles per CTA."""
    assert _plan(ctx, "wgrad", shape)["kind"] == "wgrad-runs"


def test_clusters_have_their_sms_to_themselves(ctx):
    """CTAs that wait for one another must not share an SM with CTAs of another cluster (their TMEM allocations could wait in a circle):
    each takes more than half of an SM's 228 KB of shared memory, also where the plan needs less."""
    rng = random.Random(1)
    clusters = raised = 0
    for _ in range(1500):
        hw = rng.choice([4, 8, 16, 32])
        shape = (rng.randint(1, 600), hw, hw, 16 * rng.randint(1, 40), 16 * rng.randint(1, 40), rng.choice([1, 3]), rng.choice([1, 1, 2]))
        for which in ("fwd", "dgrad"):
            plan = _plan(ctx, which, shape)
            if plan["pair"] or plan["splits"] > 1:
                clusters += 1
                raised += plan["smem_bytes"] == 115 * 1024
                assert plan["smem_bytes"] > 114 * 1024, (shape, plan)
    assert clusters >= 200 and raised >= 5, (clusters, raised)


def test_plan_of_a_call_with_sums(ctx):
    """256-channel tiles whose MMAs hide the epilogue work in blocks only where they take sums: the query tells both apart, and the
    shared memory that it reports holds the blocks."""
    from paper_2503_23186_b200 import binding
    d = binding.conv_desc(1024, 8, 8, 256, 256, 3, 1)
    plain, sums = ctx.conv2d_plan(d, "fwd"), ctx.conv2d_plan(d, "fwd", sums=True)
    assert plain["block_cols"] == 0 and sums["block_cols"] == 64, (plain, sums)
    assert sums["smem_bytes"] == plain["smem_bytes"] + 24 * 1024
    for which in ("dgrad", "wgrad"):
        with pytest.raises(binding.B2CError):
            ctx.conv2d_plan(d, which, sums=True)


# 256-channel outputs of 1024 images: 3x3 layers whose ring leaves no room for the epilogue's blocks take the statistics in a pass of their own
@pytest.mark.parametrize("c,r,blocks", [(64, 3, False), (64, 1, True), (128, 1, True)])
def test_statistics_in_the_epilogue_where_it_works_in_blocks(ctx, c, r, blocks):
    from paper_2503_23186_b200 import binding, workloads as wl
    n, hw, k = 1024, 16, 256
    plan = ctx.conv2d_plan(binding.conv_desc(n, hw, hw, c, k, r, 1), "fwd", sums=True)
    assert (plan["block_cols"] != 0) == blocks, plan
    spec = [dict(kind="conv", src=0, C=16, K=c, R=1, stride=1, pad=0, H=hw, W=hw, name="c0"), dict(kind="bn", src=1, C=c, H=hw, W=hw, relu=True, res=-1, name="b0"),
            dict(kind="conv", src=2, C=c, K=k, R=r, stride=1, pad=r // 2, H=hw, W=hw, name="c1"), dict(kind="bn", src=3, C=k, H=hw, W=hw, relu=True, res=-1, name="b1"),
            dict(kind="avgpool", src=4, C=k, H=hw, W=hw, name="pool"), dict(kind="fc", src=5, C=k, K=10, name="fc"), dict(kind="xent", src=6, K=10, name="xent")]
    net = binding.Net(ctx, spec, n)
    net.load_params(wl.init_params(spec, 1))
    net.profile_read()
    net.train_step(torch.zeros((n, hw, hw, 16), dtype=torch.bfloat16, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda"), 1, 0.1, 0.9, 0.0, update=False)
    assert ctx.device_status() == 0
    _, launches = net.profile_read()
    assert launches["bn_fwd"] == (2 if blocks else 3), launches   # an apply pass each, and the statistics' own
    net.close()


# x tiles of 3x3 weight gradients: half of the widest where the sending of partial sums is most of the launch; not where half the width makes a
# second wave of a few CTAs, or gives up equal runs
@pytest.mark.parametrize("shape,tile,kind", [
    ((50, 16, 16, 128, 128, 3, 1), 64, "wgrad"), ((128, 8, 8, 256, 512, 3, 2), 64, "wgrad"), ((600, 16, 16, 128, 128, 3, 1), 128, "wgrad"),
    ((9, 32, 32, 256, 16, 3, 2), 128, "wgrad"), ((14, 32, 32, 160, 16, 3, 2), 160, "wgrad"), ((10, 8, 8, 640, 16, 3, 2), 64, "wgrad"),   # 16 output channels
    ((8, 8, 8, 640, 640, 3, 1), 128, "wgrad"), ((24, 32, 32, 512, 640, 3, 1), 128, "wgrad-runs"), ((228, 8, 8, 1024, 640, 3, 1), 128, "wgrad")],
    ids=lambda v: "n{}h{}w{}c{}k{}r{}s{}".format(*v) if isinstance(v, tuple) else str(v))
def test_tile_width_of_weight_gradients(ctx, shape, tile, kind):
    plan = _plan(ctx, "wgrad", shape)
    assert plan["tile_channels"] == tile and plan["kind"] == kind, plan


@pytest.mark.parametrize("shape,plain,sums", [((60, 32, 32, 608, 64, 3, 1), 0, 0), ((150, 32, 32, 224, 64, 3, 1), 0, 0), ((200, 32, 32, 160, 64, 3, 1), 32, 32),
                                              ((500, 32, 32, 32, 64, 3, 1), 0, 32), ((300, 32, 32, 48, 64, 3, 1), 32, 32), ((500, 32, 32, 32, 64, 1, 1), 32, 32), ((4, 64, 64, 32, 64, 3, 1), 32, 32)],
                         ids=lambda v: "n{}h{}w{}c{}k{}r{}s{}".format(*v) if isinstance(v, tuple) else str(v))
def test_blocks_where_the_mmas_hide_the_epilogue(ctx, shape, plain, sums):
    from paper_2503_23186_b200 import binding
    d = binding.conv_desc(*shape)
    assert (ctx.conv2d_plan(d, "fwd")["block_cols"], ctx.conv2d_plan(d, "fwd", sums=True)["block_cols"]) == (plain, sums)
