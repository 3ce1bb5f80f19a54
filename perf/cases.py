"""The work a user of this library has it do, as timed cases.

`listed()` names the cases, `draw(rng)` gives more of the same ranges, `prepare` makes what a program has in hand
before the call, `run` makes one pass through the public entry points, `work` counts what a pass cannot do without
and `tolerance` states how far two correct implementations of the same precision may lie apart.

Kinds of case:
  step    one optimiser step over a layer list (`binding.Net.train_step`): forward, loss, backward, update.
  conv    one convolution layer on its own: forward with BatchNorm sums, data gradient, weight gradient.
  block   one residual basic block, forward and backward, through the single-operation entry points.
  bn      BatchNorm(+residual)+ReLU forward and backward on its own.
  update  gradient average + SGD-momentum update of a replica after the exchange of the gradient sums.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_23186_b200 import binding, workloads as wl

# momentum and weight decay as everywhere in this repository; the learning rate is that of a late stage of training: the
# gradients of a deep BatchNorm net differ by tens of percent between two runs (sums in an unspecified order, amplified
# layer by layer), and a small step keeps the weights of successive passes comparable
LR, MU, WD, EPS = 0.01, 0.9, 5e-4, 1e-5


def listed():
    return [
        # the library's main configuration: a batch of 1024 as eight micro-batches side by side in one pass
        dict(name="step_resnet18_b1024", kind="step", net="resnet18", micro_batch=128, n_micro=8, concurrent=8),
        # the same net at a small batch, where launches and latency count
        dict(name="step_resnet18_b128", kind="step", net="resnet18", micro_batch=128, n_micro=1, concurrent=1),
        # gradient accumulation under a memory limit: micro-batches of an odd size, one after the other
        dict(name="step_resnet18_4x50", kind="step", net="resnet18", micro_batch=50, n_micro=4, concurrent=1),
        # wide channels that are multiples of 160
        dict(name="step_wrn28_10_b256", kind="step", net="wrn28_10", micro_batch=256, n_micro=1, concurrent=1),
        # the largest: bottleneck blocks, many 1x1 layers, up to 2048 channels
        dict(name="step_resnet50_b1024", kind="step", net="resnet50", micro_batch=128, n_micro=8, concurrent=8),
        # a first experiment: a few layers on 16x16 images, bound by latency
        dict(name="step_small_b16", kind="step", net="residual", stem=64, width=64, stages=2, blocks=1, hw=16, classes=10, micro_batch=16,
             n_micro=1, concurrent=1),
        # the smallest layer: 16 channels, eight images
        dict(name="conv_16_16_b8", kind="conv", n=8, hw=32, c=16, k=16, r=3, stride=1),
        # a layer that halves the image, at a batch that fills no tile evenly
        dict(name="conv_128_256_s2_b250", kind="conv", n=250, hw=16, c=128, k=256, r=3, stride=2),
        # one basic block of the first stage on its own
        dict(name="block_64_b128", kind="block", n=128, hw=32, c=64),
        # normalisation behind the widening 1x1 layer of a bottleneck block, with its shortcut
        dict(name="bn_256_res_b128", kind="bn", n=128, hw=32, c=256, res=True, mask=True, running=True),
        # a data-parallel replica's update once the gradients have been summed over the replicas
        dict(name="update_resnet50", kind="update", net="resnet50", n_avg=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi):
    """A channel count: a multiple of 16, the usual widths among them."""
    if rng.random() < 0.5:
        return rng.choice([w for w in (16, 32, 64, 128, 160, 256, 320, 512, 640, 1024, 2048) if lo <= w <= hi])
    return max(lo, _log(rng, lo, hi) // 16 * 16)


# what a drawn case may cost at most, as shares of the largest listed one
_MAX_FLOPS = 7.9e12
_MAX_BYTES = 2.0e10   # activations of one pass


def draw(rng):
    kind = rng.choice(["step", "step", "step", "conv", "conv", "block", "bn", "update"])
    if kind == "step":
        case = dict(kind="step")
        net = rng.choice(["resnet18", "wrn28_10", "resnet50", "residual", "residual", "bottleneck"])
        case["net"] = net
        if net in ("residual", "bottleneck"):
            case.update(stem=rng.choice([16, 32, 64]), width=rng.choice([16, 32, 48, 64, 96, 128]), stages=rng.choice([1, 2, 3]),
                        blocks=rng.choice([1, 2]), hw=rng.choice([16, 32]), classes=rng.choice([10, 100]))
        case["micro_batch"] = _log(rng, 8, 256)
        case["n_micro"] = rng.choice([1, 1, 2, 4, 8])
        case["concurrent"] = rng.choice([1, case["n_micro"]])
        while case["micro_batch"] > 1 and (work(case)["flops"] > _MAX_FLOPS or _activation_bytes(case) > _MAX_BYTES):
            case["micro_batch"] = case["micro_batch"] * 2 // 3
        return case
    if kind == "conv":
        case = dict(kind="conv", n=_log(rng, 4, 1024), hw=rng.choice([4, 8, 16, 32]), c=_channels(rng, 16, 640), k=_channels(rng, 16, 640),
                    r=rng.choice([3, 3, 1]), stride=rng.choice([1, 1, 2]))
        while case["n"] > 1 and work(case)["flops"] > _MAX_FLOPS / 4:
            case["n"] //= 2
        return case
    if kind == "block":
        case = dict(kind="block", n=_log(rng, 4, 512), hw=rng.choice([8, 16, 32]), c=_channels(rng, 64, 512))
        while case["n"] > 1 and work(case)["flops"] > _MAX_FLOPS / 4:
            case["n"] //= 2
        return case
    if kind == "bn":
        case = dict(kind="bn", n=_log(rng, 4, 1024), hw=rng.choice([4, 8, 16, 32]), c=_channels(rng, 16, 2048), res=rng.random() < 0.5,
                    mask=rng.random() < 0.7, running=rng.random() < 0.5)
        while case["n"] > 1 and work(case)["bytes"] > _MAX_BYTES / 4:
            case["n"] //= 2
        return case
    net = rng.choice(["resnet18", "wrn28_10", "resnet50", "residual"])
    case = dict(kind="update", net=net, n_avg=_log(rng, 1, 64))
    if net == "residual":
        case.update(stem=rng.choice([16, 32, 64]), width=rng.choice([32, 48, 64, 96, 128, 160]), stages=rng.choice([2, 3, 4]), blocks=rng.choice([1, 2, 3]), hw=32,
                    classes=rng.choice([10, 100]))
    return case


# ------------------------------------------------------------------------------------------
# layer lists
# ------------------------------------------------------------------------------------------
def _spec(case):
    net = case["net"]
    if net == "resnet18":
        return wl.resnet18_spec()
    if net == "wrn28_10":
        return wl.wrn28_10_spec()
    if net == "resnet50":
        return wl.resnet50_spec()
    widths = [case["width"] << i for i in range(case["stages"])]
    strides = [1] + [2] * (case["stages"] - 1)
    if net == "residual":
        return wl.residual_net_spec(case["stem"], widths, strides, case["blocks"], case["classes"], image_hw=case["hw"])
    return wl.bottleneck_net_spec(case["stem"], widths, strides, [case["blocks"]] * case["stages"], case["classes"], image_hw=case["hw"])


def _params(spec):
    n = 0
    for L in spec:
        if L["kind"] == "conv":
            n += L["K"] * L["R"] ** 2 * L["C"]
        elif L["kind"] == "bn":
            n += 2 * L["C"]
        elif L["kind"] == "fc":
            n += L["K"] * L["C"] + L["K"]
    return n


def _activation_bytes(case):
    """Layer outputs and their gradients of one pass of a step."""
    n = case["micro_batch"] * case["concurrent"]
    e = sum(L["H"] // L.get("stride", 1) * (L["W"] // L.get("stride", 1)) * L.get("K", L["C"]) for L in _spec(case) if L["kind"] in ("conv", "bn"))
    return 4.0 * n * e


def _conv_flops(n, hw, c, k, r, stride):
    return 2.0 * n * (hw // stride) ** 2 * k * r * r * c


def work(case):
    """Bytes (each input once, each output once) and floating-point operations of one pass."""
    kind = case["kind"]
    if kind == "step":
        spec = _spec(case)
        images = case["micro_batch"] * case["n_micro"]
        flops = 0.0
        for L in spec:
            if L["kind"] == "conv":   # forward, weight gradient and, except for the first layer, data gradient
                flops += (3 if L["src"] != 0 else 2) * _conv_flops(images, L["H"], L["C"], L["K"], L["R"], L["stride"])
            elif L["kind"] == "fc":
                flops += 3 * 2.0 * images * L["C"] * L["K"]
        hw, c = spec[0]["H"], spec[0]["C"]
        return {"bytes": images * (2.0 * hw * hw * c + 4.0) + 16.0 * _params(spec), "flops": flops}
    if kind == "conv":
        n, hw, c, k, r, st = (case[f] for f in ("n", "hw", "c", "k", "r", "stride"))
        x, y, w = 2.0 * n * hw * hw * c, 2.0 * n * (hw // st) ** 2 * k, 2.0 * k * r * r * c
        return {"bytes": 2 * x + 2 * y + 2 * w + 2 * w, "flops": 3 * _conv_flops(n, hw, c, k, r, st)}   # x, y, dy, dx, both filter copies, fp32 dw
    if kind == "block":
        n, hw, c = case["n"], case["hw"], case["c"]
        e, w = 2.0 * n * hw * hw * c, 2.0 * 9 * c * c
        return {"bytes": 5 * e + 2 * 4 * w, "flops": 6 * _conv_flops(n, hw, c, c, 3, 1)}   # x, out, upstream gradient, dx, shortcut gradient
    if kind == "bn":
        e = 2.0 * case["n"] * case["hw"] ** 2 * case["c"]
        res = 1 if case["res"] else 0
        # forward: y (+ residual) in, a out; backward: upstream gradient in, dy (+ shortcut gradient) out
        return {"bytes": e * (4 + 2 * res), "flops": 20.0 * e / 2}
    p = _params(_spec(case))
    return {"bytes": 28.0 * p, "flops": 6.0 * p}   # w, v, g read; w, v, g = 0 and both bf16 copies written


def tolerance(case):
    """About four times what two runs, and a run with the sums in another order, were seen to lie apart."""
    kind = case["kind"]
    if kind == "step":
        # two passes of one state: loss 2e-3, weights 3e-3 (a single weight 0.25 of their root mean square) on the deepest
        # net; momentum of the shallow ones 8e-3
        return {"rel": 1e-2 if not _shallow(case) else 3e-2, "max": 0.9}
    if kind == "conv":
        return {"rel": 3e-4, "max": 0.03}   # bf16 results one step apart in 1e-3 of the places; fp32 sums 1e-7
    if kind == "block":
        return {"rel": 8e-3, "max": 0.9}    # where a sum falls on the other side of a ReLU's zero, a whole gradient appears
    if kind == "bn":
        return {"rel": 1e-4, "max": 0.03}
    return {"rel": 1e-5, "max": 0.01}       # fp32 update: 1e-7; bf16 copies one step apart in few places


def _shallow(case):
    """Nets of one or two blocks: their gradients (the momentum after a step) are comparable between two runs."""
    return case["kind"] == "step" and case["net"] in ("residual", "bottleneck") and case["stages"] * case["blocks"] <= 2


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
class _Draws:
    """Seeded normal and integer tensors, made on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed))

    def normal(self, shape, std=1.0, dtype=torch.bfloat16):
        return (torch.randn(shape, generator=self.gen, device="cuda") * std).to(dtype)

    def labels(self, n, classes):
        return torch.randint(0, classes, (n,), generator=self.gen, device="cuda", dtype=torch.int32)


def _f32(n):
    return torch.empty(n, dtype=torch.float32, device="cuda")


def prepare(case, seed):
    draws = _Draws(seed)
    return {"step": _prepare_step, "conv": _prepare_conv, "block": _prepare_block, "bn": _prepare_bn, "update": _prepare_update}[case["kind"]](case, seed, draws)


def run(state):
    return state["run"](state)


# ---- step
def _prepare_step(case, seed, draws):
    spec = _spec(case)
    ctx = binding.Context(torch.cuda.current_device())
    net = binding.Net(ctx, spec, case["micro_batch"], n_concurrent=case["concurrent"])
    net.load_params(wl.init_params(spec, seed))
    n, hw, c = case["micro_batch"] * case["n_micro"], spec[0]["H"], spec[0]["C"]
    images = draws.normal((n, hw, hw, c))
    labels = draws.labels(n, spec[-1]["K"])
    return dict(run=_run_step, ctx=ctx, net=net, images=images, labels=labels, n_micro=case["n_micro"], momentum=_shallow(case))


def _run_step(s):
    net = s["net"]
    loss = net.train_step(s["images"], s["labels"], s["n_micro"], LR, MU, WD)
    return {"loss": loss, "w": net.w, "v": net.v} if s["momentum"] else {"loss": loss, "w": net.w}


# ---- one convolution layer
def _packed(ctx, w, k, rs, c):
    """The data-gradient layout of a filter bank, as a program refreshes it once per update."""
    out = torch.empty_like(w)
    ctx.weight_pack_dgrad([(0, k, rs, c)], w.reshape(-1), out.reshape(-1))
    return out


def _prepare_conv(case, seed, draws):
    n, hw, c, k, r, st = (case[f] for f in ("n", "hw", "c", "k", "r", "stride"))
    ctx = binding.Context(torch.cuda.current_device())
    x = draws.normal((n, hw, hw, c))
    w = draws.normal((k, r, r, c), std=math.sqrt(2.0 / (r * r * c)))
    g = draws.normal((n, hw // st, hw // st, k))
    return dict(run=_run_conv, ctx=ctx, d=binding.conv_desc(n, hw, hw, c, k, r, st), x=x, w=w, w_dgrad=_packed(ctx, w, k, r * r, c), g=g, y=torch.empty_like(g),
                stats=torch.zeros(2 * k, dtype=torch.float64, device="cuda"), dx=torch.empty_like(x), dw=_f32(k * r * r * c).view(k, r, r, c))


def _run_conv(s):
    ctx, d = s["ctx"], s["d"]
    s["stats"].zero_()
    ctx.conv2d_fwd(d, s["x"], s["w"], s["y"], ch_stats=s["stats"])
    ctx.conv2d_dgrad(d, s["g"], s["w_dgrad"], s["dx"])
    ctx.conv2d_wgrad(d, s["g"], s["x"], s["dw"])
    return {k: s[k] for k in ("y", "stats", "dx", "dw")}


# ---- one basic block: out = relu(bn(conv(relu(bn(conv(x))))) + x)
def _prepare_block(case, seed, draws):
    n, hw, c = case["n"], case["hw"], case["c"]
    ctx = binding.Context(torch.cuda.current_device())
    s = dict(run=_run_block, ctx=ctx, d=binding.conv_desc(n, hw, hw, c, c, 3, 1), n=n, hw=hw, c=c)
    s["x"], s["g"] = draws.normal((n, hw, hw, c)), draws.normal((n, hw, hw, c))
    for i in (1, 2):
        s[f"w{i}"] = draws.normal((c, 3, 3, c), std=math.sqrt(2.0 / (9 * c)))
        s[f"wd{i}"] = _packed(ctx, s[f"w{i}"], c, 9, c)
        s[f"gamma{i}"] = 1.0 + draws.normal((c,), 0.1, torch.float32)
        s[f"beta{i}"] = draws.normal((c,), 0.1, torch.float32)
        s[f"mask{i}"] = torch.empty(n * hw * hw * c // 8, dtype=torch.uint8, device="cuda")
        s[f"dw{i}"] = _f32(9 * c * c).view(c, 3, 3, c)
        for name in ("mean", "invstd", "dgamma", "dbeta"):
            s[f"{name}{i}"] = _f32(c)
    for name in ("y1", "a1", "y2", "out", "dy2", "dres", "da1", "dy1", "dx"):
        s[name] = torch.empty_like(s["x"])
    s["stats"] = torch.zeros((2, 2 * c), dtype=torch.float64, device="cuda")
    s["ws"] = torch.empty(binding.Context.bn_relu_bwd_workspace_bytes(c), dtype=torch.uint8, device="cuda")
    return s


def _run_block(s):
    ctx, d, n, hw, c = s["ctx"], s["d"], s["n"], s["hw"], s["c"]
    s["stats"].zero_()
    ctx.conv2d_fwd(d, s["x"], s["w1"], s["y1"], ch_stats=s["stats"][0])
    ctx.bn_relu_fwd(n, hw, hw, c, s["y1"], s["stats"][0], True, s["gamma1"], s["beta1"], None, True, EPS, s["a1"], s["mean1"], s["invstd1"], relu_mask=s["mask1"])
    ctx.conv2d_fwd(d, s["a1"], s["w2"], s["y2"], ch_stats=s["stats"][1])
    ctx.bn_relu_fwd(n, hw, hw, c, s["y2"], s["stats"][1], True, s["gamma2"], s["beta2"], s["x"], True, EPS, s["out"], s["mean2"], s["invstd2"],
                    relu_mask=s["mask2"])
    ctx.bn_relu_bwd(n, hw, hw, c, s["g"], None, s["y2"], s["out"], s["gamma2"], s["mean2"], s["invstd2"], True, s["dy2"], s["dres"], s["dgamma2"], s["dbeta2"],
                    False, s["ws"], relu_mask=s["mask2"])
    ctx.conv2d_wgrad(d, s["dy2"], s["a1"], s["dw2"])
    ctx.conv2d_dgrad(d, s["dy2"], s["wd2"], s["da1"])
    ctx.bn_relu_bwd(n, hw, hw, c, s["da1"], None, s["y1"], s["a1"], s["gamma1"], s["mean1"], s["invstd1"], True, s["dy1"], None, s["dgamma1"], s["dbeta1"],
                    False, s["ws"], relu_mask=s["mask1"])
    ctx.conv2d_wgrad(d, s["dy1"], s["x"], s["dw1"])
    ctx.conv2d_dgrad(d, s["dy1"], s["wd1"], s["dx"])
    # (the shortcut's gradient is the masked upstream gradient: `bn` compares it)
    return {k: s[k] for k in ("out", "dx", "dw1", "dw2", "dgamma1", "dbeta1", "dgamma2", "dbeta2", "mean1", "invstd1", "mean2", "invstd2")}


# ---- BatchNorm (+ residual) + ReLU
def _prepare_bn(case, seed, draws):
    n, hw, c = case["n"], case["hw"], case["c"]
    shape = (n, hw, hw, c)
    s = dict(run=_run_bn, ctx=binding.Context(torch.cuda.current_device()), n=n, hw=hw, c=c)
    s["y"] = draws.normal(shape, 1.5) + draws.normal((c,), 0.5)   # channels with means of their own
    s["da"] = draws.normal(shape, 1e-3)
    s["res"] = draws.normal(shape) if case["res"] else None
    s["gamma"], s["beta"] = 1.0 + draws.normal((c,), 0.1, torch.float32), draws.normal((c,), 0.1, torch.float32)
    s["a"], s["dy"] = torch.empty_like(s["y"]), torch.empty_like(s["y"])
    s["dres"] = torch.empty_like(s["y"]) if case["res"] else None
    s["mask"] = torch.empty(n * hw * hw * c // 8, dtype=torch.uint8, device="cuda") if case["mask"] else None
    s["stats"] = torch.zeros(2 * c, dtype=torch.float64, device="cuda")
    for name in ("mean", "invstd", "dgamma", "dbeta"):
        s[name] = _f32(c)
    s["run_mean"], s["run_var"] = (torch.zeros(c, device="cuda"), torch.ones(c, device="cuda")) if case["running"] else (None, None)
    s["ws"] = torch.empty(binding.Context.bn_relu_bwd_workspace_bytes(c), dtype=torch.uint8, device="cuda")
    return s


def _run_bn(s):
    ctx, n, hw, c = s["ctx"], s["n"], s["hw"], s["c"]
    ctx.bn_relu_fwd(n, hw, hw, c, s["y"], s["stats"], False, s["gamma"], s["beta"], s["res"], True, EPS, s["a"], s["mean"], s["invstd"], s["run_mean"], s["run_var"],
                    0.1, relu_mask=s["mask"])
    ctx.bn_relu_bwd(n, hw, hw, c, s["da"], None, s["y"], s["a"], s["gamma"], s["mean"], s["invstd"], True, s["dy"], s["dres"], s["dgamma"], s["dbeta"], False,
                    s["ws"], relu_mask=s["mask"])
    return {k: s[k] for k in ("a", "dy", "dres", "dgamma", "dbeta", "mean", "invstd", "run_mean", "run_var") if s[k] is not None}


# ---- update of a replica
def _prepare_update(case, seed, draws):
    spec = _spec(case)
    ctx = binding.Context(torch.cuda.current_device())
    net = binding.Net(ctx, spec, 1)
    params = wl.init_params(spec, seed)
    net.load_params(params)
    # gradient sums as the exchange leaves them; the arrays' padding holds zeros, as after a backward pass
    net.g.copy_(draws.normal((net.param_count,), 1e-2, torch.float32))
    net.v.copy_(draws.normal((net.param_count,), 1e-2, torch.float32))
    if net.param_count != _params(spec):
        real = torch.from_numpy(net.pack({k: np.ones_like(v) for k, v in params.items()})).cuda()
        net.g.mul_(real)
        net.v.mul_(real)
    return dict(run=_run_update, ctx=ctx, net=net, n_avg=case["n_avg"])


def _run_update(s):
    net = s["net"]
    net.apply_update(s["n_avg"], LR, MU, WD)
    return {"w": net.w, "v": net.v, "w_bf16": net.w_bf16, "w_dgrad": net.w_dgrad}
