"""Launches that start beside the one before them (data gradients behind weight gradients, shortcut convolutions behind a
BatchNorm): every tensor of a chain without BatchNorm bit for bit against the same passes with the launches one after the other, every layer
of nets with shortcuts against the oracle on its own device inputs, and as a rough check the gradient sums of many passes."""
import numpy as np
import pytest
import torch

from netcheck import _shape, check_step, grad_slots
from paper_2503_23186_b200 import workloads as wl
from parity import dev_bf16

pytestmark = pytest.mark.gpu


def _gradients(spec, micro_batch, n_micro, concurrent, passes, monkeypatch, pdl):
    from paper_2503_23186_b200 import binding
    monkeypatch.setenv("B2C_PDL", pdl)
    ctx = binding.Context(0)
    net = binding.Net(ctx, spec, micro_batch, n_concurrent=concurrent)
    net.load_params(wl.perturb_bn_params(wl.init_params(spec, 3), 3))
    hw, c, classes = spec[0]["H"], spec[0]["C"], spec[-1]["K"]
    losses, total = [], None
    for i in range(passes):   # other images every time: a gradient computed from the previous pass's tensors shows
        images, labels = wl.image_batch(10 + i, micro_batch * n_micro, hw=hw, c=c, classes=classes)
        loss = net.train_step(torch.from_numpy(images).to(torch.bfloat16).cuda(), torch.from_numpy(labels).cuda(), n_micro, 0.1, 0.9, 5e-4, update=False)
        losses.append(loss.clone())
    assert ctx.device_status() == 0
    total = net.unpack(net.g)
    net.close()
    ctx.close()
    return [x.item() for x in losses], total


@pytest.mark.parametrize("case", [("residual", 24, 3, 1), ("residual", 32, 2, 2), ("bottleneck", 8, 4, 1)], ids=lambda c: "{}-{}x{}-{}".format(*c))
def test_overlapping_launches_give_the_same_gradients(case, monkeypatch):
    net, micro_batch, n_micro, concurrent = case
    spec = (wl.residual_net_spec(32, (32, 64), (1, 2), 1, 10, image_hw=16) if net == "residual"
            else wl.bottleneck_net_spec(16, (16, 32), (1, 2), (1, 1), 10, image_hw=16))
    got_loss, got = _gradients(spec, micro_batch, n_micro, concurrent, 6, monkeypatch, "1")
    want_loss, want = _gradients(spec, micro_batch, n_micro, concurrent, 6, monkeypatch, "0")
    np.testing.assert_allclose(got_loss, want_loss, rtol=2e-3)
    for name in want:
        # two correct runs of a net of one or two blocks lie up to 3e-2 apart (sums in another order move ReLU signs): this shows tensors that were
        # read too early as a whole, the tests below parts of them
        err = np.linalg.norm(got[name] - want[name]) / np.linalg.norm(want[name])
        assert err < 0.1, (name, err)


def _chain(hw=16):
    """Convolutions straight behind one another: nothing in their tensors depends on an order of sums."""
    spec, h = [], hw
    for i, (c, k, r, st) in enumerate([(16, 64, 3, 1), (64, 64, 3, 1), (64, 128, 3, 2), (128, 64, 1, 1), (64, 64, 3, 1), (64, 96, 1, 2), (96, 128, 3, 1)]):
        spec.append(dict(kind="conv", src=len(spec), C=c, K=k, R=r, stride=st, pad=r // 2, H=h, W=h, name=f"c{i}"))
        h //= st
    spec.append(dict(kind="avgpool", src=len(spec), C=128, H=h, W=h, name="pool"))
    spec.append(dict(kind="fc", src=len(spec), C=128, K=10, name="fc"))
    spec.append(dict(kind="xent", src=len(spec), K=10, name="xent"))
    return spec


def _passes(spec, micro_batch, pdl, split_k, passes, monkeypatch):
    from paper_2503_23186_b200 import binding
    monkeypatch.setenv("B2C_PDL", pdl)
    monkeypatch.setenv("B2C_SPLIT_K", split_k)
    ctx = binding.Context(0)
    for L in spec:
        if L["kind"] == "conv":
            for which in ("fwd", "dgrad"):
                kind = ctx.conv2d_plan(binding.conv_desc(micro_batch, L["H"], L["W"], L["C"], L["K"], L["R"], L["stride"]), which)["kind"]
                assert kind != "shared-units" and (kind != "one-wave" or split_k == "1"), (L, kind)
    net = binding.Net(ctx, spec, micro_batch)
    net.load_params(wl.init_params(spec, 3))
    _, contributions = grad_slots(spec)
    seen = []
    for i in range(passes):   # other images every time: what is read from the pass before shows
        images, labels = wl.image_batch(40 + i, micro_batch, hw=16, c=16, classes=10)
        net.train_step(dev_bf16(images), torch.from_numpy(labels).cuda(), 1, 0.1, 0.9, 0.0, update=False)
        for t in range(1, len(spec)):
            shape = _shape(spec, t, micro_batch, net)
            seen.append((i, t, "out", net.tensor_view(t, shape, torch.float32 if spec[t - 1]["kind"] == "fc" else torch.bfloat16).clone()))
            seen += [(i, t, "gradient", net.tensor_view(t, shape, torch.bfloat16, True, slot).clone()) for slot in range(contributions[t])]
    assert ctx.device_status() == 0
    weights = net.unpack(net.g)
    net.close()
    ctx.close()
    return seen, weights


@pytest.mark.parametrize("split_k", ["1", "0"], ids=["one-wave", "persistent"])
@pytest.mark.parametrize("micro_batch", [24, 200])
def test_overlapping_launches_give_the_same_bits(micro_batch, split_k, monkeypatch):
    spec = _chain()
    got, got_w = _passes(spec, micro_batch, "1", split_k, 8, monkeypatch)
    want, want_w = _passes(spec, micro_batch, "0", split_k, 8, monkeypatch)
    for (i, t, what, a), (_, _, _, b) in zip(got, want):
        assert bool(torch.isfinite(b.float()).all()) and torch.equal(a, b), (i, t, what, int((a != b).sum()))
    for name in want_w:   # sums of fp32 partial sums in any order: a few 2^-24 of the largest partial sums
        assert np.linalg.norm(got_w[name] - want_w[name]) <= 1e-5 * np.linalg.norm(want_w[name]), name


@pytest.mark.parametrize("split_k", ["1", "0"], ids=["one-wave", "persistent"])
@pytest.mark.parametrize("net_kind", ["residual", "bottleneck"])
def test_layers_of_overlapping_passes(net_kind, split_k, monkeypatch):
    """Nets whose stages begin with a stride-2 shortcut: after several passes over other images, every layer of the last one."""
    from paper_2503_23186_b200 import binding
    monkeypatch.setenv("B2C_SPLIT_K", split_k)
    spec = (wl.residual_net_spec(32, (32, 64), (1, 2), 1, 10, image_hw=16, image_c=16) if net_kind == "residual"
            else wl.bottleneck_net_spec(16, (16, 32), (1, 2), (1, 1), 10, image_hw=16, image_c=16))
    ctx = binding.Context(0)
    try:
        net = binding.Net(ctx, spec, 12)
        net.load_params(wl.perturb_bn_params(wl.init_params(spec, 3), 3))
        for check in range(3):
            batches = [wl.image_batch(70 + 10 * check + i, 12, hw=16, c=16, classes=10) for i in range(5)]
            device = [(dev_bf16(x), torch.from_numpy(y).cuda()) for x, y in batches]
            for x, y in device[:-1]:
                net.train_step(x, y, 1, 0.1, 0.9, 0.0, update=False)
            net.g.zero_()
            net.train_step(*device[-1], 1, 0.1, 0.9, 0.0, update=False)
            assert ctx.device_status() == 0
            check_step(net, spec, *batches[-1], 12).assert_ok()
        net.close()
    finally:
        ctx.close()
