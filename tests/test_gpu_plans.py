"""Which kernel a convolution layer gets: the rules of the planner at layers where a wrong estimate costs much."""
import random

import pytest

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
