"""The one-pass update of a network (average, momentum, weight decay, both bf16 copies) and the transposed layout alone."""
import numpy as np
import pytest
import torch

import oracle
from paper_2503_23186_b200 import workloads as wl
from parity import dev_bf16

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2503_23186_b200 import binding
    c = binding.Context(0)
    yield c
    assert c.device_status() == 0
    c.close()


def _flipped(w):   # [k][rs][c] -> [c][rs - 1 - t][k]
    return np.ascontiguousarray(np.transpose(w, (2, 1, 0))[:, ::-1])


# tiles of 64 x 64 filled, with remainders of 16 and 48 in either direction, and smaller than one
@pytest.mark.parametrize("width,stages", [(16, 1), (48, 2), (160, 1)])
def test_net_update_and_transposed_copy(ctx, width, stages):
    from paper_2503_23186_b200 import binding
    spec = wl.residual_net_spec(16, [width << i for i in range(stages)], [1, 2][:stages], 1, 10, image_hw=8)
    net = binding.Net(ctx, spec, 4)
    params = wl.init_params(spec, 50)
    net.load_params(params)
    r = wl.rng_for(50, "update")
    v0 = {k: (0.01 * r.standard_normal(p.shape)).astype(np.float32) for k, p in params.items()}
    g0 = {k: r.standard_normal(p.shape).astype(np.float32) for k, p in params.items()}
    net.v.copy_(torch.from_numpy(net.pack(v0)))
    net.g.copy_(torch.from_numpy(net.pack(g0)))
    net.apply_update(3, 0.1, 0.9, 5e-4)
    assert ctx.device_status() == 0
    w, v = net.unpack(net.w), net.unpack(net.v)
    for name, p in params.items():   # fp32 arithmetic on identical inputs: a few roundings of 6e-8
        rw, rv = oracle.sgd_momentum(p, v0[name], g0[name], 1.0 / 3, 0.1, 0.9, 5e-4)
        assert np.max(np.abs(w[name] - rw)) <= 1e-6 * max(np.max(np.abs(rw)), 1e-3), name
        assert np.max(np.abs(v[name] - rv)) <= 1e-6 * max(np.max(np.abs(rv)), 1e-3), name
    assert torch.count_nonzero(net.g).item() == 0
    assert torch.equal(net.w_bf16, net.w.to(torch.bfloat16))
    bf, dg = net.w_bf16.float().cpu().numpy(), net.w_dgrad.float().cpu().numpy()
    ranges = net.weight_layer_ranges()
    layers = [L for L in spec if L["kind"] in ("conv", "fc")]
    for i, (L, (b, e)) in enumerate(zip(layers, ranges)):
        rs = L["R"] ** 2 if L["kind"] == "conv" and i > 0 else 1   # the first convolution is stored as rows of the patch matrix
        k = L["K"] if L["kind"] == "conv" else -(-L["K"] // 64) * 64
        assert np.array_equal(dg[b:e].reshape(-1, rs, k), _flipped(bf[b:e].reshape(k, rs, -1))), L["name"]
    net.close()


@pytest.mark.parametrize("k,rs,c", [(64, 9, 64), (16, 9, 16), (128, 1, 48), (72, 9, 200), (12, 9, 20), (7, 1, 5)])   # the last two: no 16-byte vectors
def test_transposed_layout(ctx, k, rs, c):
    w = wl.normal_bf16(51, f"w{k}x{c}", (k, rs, c))
    dst = torch.full((w.size + 64,), float("nan"), dtype=torch.bfloat16, device="cuda")
    ctx.weight_pack_dgrad([(0, k, rs, c)], dev_bf16(w).reshape(-1), dst)
    assert ctx.device_status() == 0
    got = dst.float().cpu().numpy()
    assert np.array_equal(got[:w.size].reshape(c, rs, k), _flipped(w)) and np.all(np.isnan(got[w.size:]))
