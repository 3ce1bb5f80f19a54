"""Weight gradients with several filter rows on M (3x3, stride 1, channel counts that leave tiles of 128 partly empty): channel blocks of 16, 32
and 64, tiles that begin and end inside a filter row, several images per chunk, images missing from the last chunk, accumulation."""
import numpy as np
import pytest
import torch

import oracle
from paper_2503_23186_b200 import workloads as wl
from parity import assert_close, dev_bf16

pytestmark = pytest.mark.gpu

SHAPES = [(17, 32, 32, 16, 16), (9, 32, 32, 64, 16), (70, 16, 16, 32, 32), (33, 16, 16, 48, 48), (67, 8, 8, 80, 80), (41, 16, 16, 16, 160), (70, 8, 8, 160, 160),
          (67, 8, 8, 64, 192), (70, 8, 8, 128, 208), (301, 4, 4, 320, 320), (1000, 4, 4, 448, 448), (1031, 2, 2, 96, 272), (5, 64, 64, 16, 48)]


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
        ctx.conv2d_wgrad(d, gd, xd, dw)
        assert ctx.device_status() == 0
        assert_close(dw, want, "dw")
        ctx.conv2d_wgrad(d, gd, xd, dw, accumulate=True)
        assert_close(dw, 2 * want, "accumulated dw")
        assert bool((flat[w.size:] == 7.0).all())
        assert np.isfinite(want).all() and ctx.device_status() == 0
    finally:
        ctx.close()
