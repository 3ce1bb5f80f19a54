"""BatchNorm sums of the backward pass taken by the one-wave data gradient: every layer of a step against the oracle on its own device inputs,
with images missing from the last tile, two gradient contributions, stride 2, a BatchNorm without ReLU, slices of 8 and 24 columns, and
several statistics groups."""
import pytest
import torch

from netcheck import check_step
from paper_2503_23186_b200 import workloads as wl
from parity import dev_bf16

pytestmark = pytest.mark.gpu


def _without_relu(c, hw):
    """conv - bn (no ReLU) - conv - bn - pool - fc: the first BatchNorm's mask does not exist."""
    spec = []
    conv = lambda src, cin, k, name: spec.append(dict(kind="conv", src=src, C=cin, K=k, R=3, stride=1, pad=1, H=hw, W=hw, name=name)) or len(spec)
    bn = lambda src, ch, relu, name: spec.append(dict(kind="bn", src=src, C=ch, H=hw, W=hw, relu=relu, res=-1, name=name)) or len(spec)
    t = conv(0, 16, c, "c0")
    t = bn(t, c, False, "bn0")
    t = conv(t, c, c, "c1")
    t = bn(t, c, True, "bn1")
    spec.append(dict(kind="avgpool", src=t, C=c, H=hw, W=hw, name="pool"))
    spec.append(dict(kind="fc", src=len(spec), C=c, K=10, name="fc"))
    spec.append(dict(kind="xent", src=len(spec), K=10, name="xent"))
    return spec


NETS = {
    "residual-48": (lambda: wl.residual_net_spec(48, (48, 96), (1, 2), 1, 10, image_hw=8, image_c=16), 5, 1),
    "residual-64": (lambda: wl.residual_net_spec(64, (64, 128), (1, 2), 2, 10, image_hw=8, image_c=3), 13, 1),
    "groups": (lambda: wl.residual_net_spec(32, (32, 64), (1, 2), 1, 10, image_hw=8, image_c=16), 8, 3),
    "bottleneck": (lambda: wl.bottleneck_net_spec(16, (16, 32), (1, 2), (2, 1), 10, image_hw=8, image_c=16), 6, 1),
    "no-relu": (lambda: _without_relu(80, 8), 3, 1),
}


@pytest.mark.parametrize("name", NETS)
def test_sums_with_the_data_gradient(name):
    from paper_2503_23186_b200 import binding
    make, micro_batch, groups = NETS[name]
    spec = make()
    hw, c = spec[0]["H"], spec[0]["C"]
    ctx = binding.Context(0)
    try:
        images, labels = wl.image_batch(61, micro_batch * groups, hw=hw, c=c, classes=10)
        net = binding.Net(ctx, spec, micro_batch, n_concurrent=groups)
        net.load_params(wl.perturb_bn_params(wl.init_params(spec, 61), 61))
        net.profile_read()
        net.train_step(dev_bf16(images), torch.from_numpy(labels).cuda(), groups, 0.1, 0.9, 5e-4, update=False)
        assert ctx.device_status() == 0
        _, launches = net.profile_read()
        assert launches["bn_bwd"] < 2 * sum(L["kind"] == "bn" for L in spec), launches   # (some took no pass of their own)
        check_step(net, spec, images, labels, micro_batch * groups, groups=groups).assert_ok()
        net.close()
    finally:
        ctx.close()


def test_stall_counters_of_launches_with_sums(monkeypatch):
    """The data gradients that take sums add their cycles to the diagnostics like the others: seven of fifteen forward and data-gradient launches."""
    from paper_2503_23186_b200 import binding
    spec = [dict(kind="conv", src=0, C=16, K=64, R=1, stride=1, pad=0, H=8, W=8, name="c0"), dict(kind="bn", src=1, C=64, H=8, W=8, relu=True, res=-1, name="b0")]
    for i in range(7):
        spec.append(dict(kind="conv", src=len(spec), C=64, K=64, R=3, stride=1, pad=1, H=8, W=8, name=f"c{i + 1}"))
        spec.append(dict(kind="bn", src=len(spec), C=64, H=8, W=8, relu=True, res=-1, name=f"b{i + 1}"))
    spec += [dict(kind="avgpool", src=len(spec), C=64, H=8, W=8, name="pool"), dict(kind="fc", src=len(spec) + 1, C=64, K=10, name="fc"),
             dict(kind="xent", src=len(spec) + 2, K=10, name="xent")]
    waited = {}
    for fuse in ("0", "1"):
        monkeypatch.setenv("B2C_FUSE_BN_BWD", fuse)
        ctx = binding.Context(0)
        net = binding.Net(ctx, spec, 16)
        net.load_params(wl.init_params(spec, 5))
        images, labels = dev_bf16(wl.image_batch(5, 16, hw=8, c=16, classes=10)[0]), torch.zeros(16, dtype=torch.int32, device="cuda")
        counters = torch.zeros(8, dtype=torch.int64, device="cuda")
        for passes in (3, 10):   # the first ones load the kernels
            net.profile_read()
            ctx.set_stall_counters(counters.zero_())
            for _ in range(passes):
                net.train_step(images, labels, 1, 0.1, 0.9, 0.0, update=False)
            assert ctx.device_status() == 0
            _, launches = net.profile_read()
        waited[fuse] = counters[3].item()   # (the weight gradient does not add to this one)
        assert (launches["bn_bwd"] < 2 * 8 * 10) == (fuse == "1"), launches
        ctx.set_stall_counters(None)
        net.close()
        ctx.close()
    assert waited["1"] > 0.8 * waited["0"], waited
