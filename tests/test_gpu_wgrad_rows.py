"""Weight gradients with several filter rows on M (3x3, stride 1, channel counts that leave tiles of 128 partly empty): channel blocks of 16, 32
and 64, tiles that begin and end inside a filter row, several images per chunk, images missing from the last chunk, accumulation."""
import pytest
import torch

import oracle
from paper_2503_23186_b200 import workloads as wl
from parity import assert_close, dev_bf16

pytestmark = pytest.mark.gpu

SHAPES = [(17, 32, 32, 16, 16), (9, 32, 32, 64, 16), (70, 16, 16, 32, 32), (33, 16, 16, 48, 48), (67, 8, 8, 80, 80), (41, 16, 16, 16, 160), (70, 8, 8, 160, 160),
          (67, 8, 8, 64, 192), (70, 8, 8, 128, 208), (301, 4, 4, 320, 320), (1000, 4, 4, 448, 448), (1031, 2, 2, 96, 272), (5, 64, 64, 16, 48),
          # blocks of 64 channels against framed x stages, one image and parts of one per chunk; several images; 16 channels
          (40, 16, 16, 64, 192), (9, 32, 32, 128, 320), (33, 16, 16, 64, 320), (300, 8, 8, 64, 192), (601, 4, 4, 64, 192), (40, 32, 32, 64, 16)]
ONE_ROW_AT_A_TIME = [(9, 32, 32, 64, 16), (67, 8, 8, 64, 192), (301, 4, 4, 320, 320)]   # the estimate finds nothing to gain


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "n{}h{}w{}c{}k{}".format(*s))
def test_filter_rows_on_m(shape):
    from paper_2503_23186_b200 import binding
    N, H, W, C, K = shape
    ctx = binding.Context(0)
    try:
        x, w, g = wl.conv_problem(71, N, H, W, C, K, 3, 1)
        want = oracle.conv2d_wgrad(g, x, 3, 3, 1, 1)
        guard = 4096
        flat = torch.full((w.size + guard,), 7.0, dtype=torch.float32, device="cuda")
        dw = flat[:w.size].view(*w.shape)
        d, gd, xd = binding.conv_desc(N, H, W, C, K, 3, 1), dev_bf16(g), dev_bf16(x)
        plan = ctx.conv2d_plan(d, "wgrad")
        block = 64 if K % 64 == 0 else 32 if K % 32 == 0 else 16
        assert plan["row_blocks"] == (0 if shape in ONE_ROW_AT_A_TIME else K // block), plan
        ctx.conv2d_wgrad(d, gd, xd, dw)
        assert ctx.device_status() == 0
        assert_close(dw, want, "dw")
        ctx.conv2d_wgrad(d, gd, xd, dw, accumulate=True)
        assert_close(dw, 2 * want, "accumulated dw")
        assert bool((flat[w.size:] == 7.0).all())
        assert ctx.device_status() == 0
    finally:
        ctx.close()
