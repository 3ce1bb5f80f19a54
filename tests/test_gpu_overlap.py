"""Launches that start beside the one before them (data gradients behind weight gradients, shortcut convolutions behind a
BatchNorm): the gradient sums of many passes against those of the same passes with the launches one after the other."""
import numpy as np
import pytest
import torch

from paper_2503_23186_b200 import workloads as wl

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
        # two correct runs of a net of one or two blocks lie up to 3e-2 apart (sums in another order move ReLU signs); a gradient that
        # was read too early, or not at all, is of the size of the gradient itself
        err = np.linalg.norm(got[name] - want[name]) / np.linalg.norm(want[name])
        assert err < 0.1, (name, err)
