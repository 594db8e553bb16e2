"""The work whose speed this library is judged by: filter gradients as training programs ask for them.

A case is one call of a public entry point (`kind`), from a single small layer, where the launches count, to
whole training steps and to feature maps of hundreds of megabytes:

  exact   gaconv_dw_exact                       the backward pass's filter gradient of one layer
  top1    gaconv_dw_approx(METHOD_TOP1)         Algorithm 1 of the paper
  topk    gaconv_dw_approx(METHOD_TOPK)         the same with several entries kept per map
  host    gaconv_dw_from_host                   inputs and result in pinned host memory, transfers included
  step    Schedule.run_step                     all layers of a network, each exact or approximated by the schedule
  train   GAConv2d forward and backward         the layer as a module of a training program

Layers come from the three CIFAR-10 networks of `layers.py`, at the batch sizes the benchmark and the schedule
sweep use, and from feature maps as image networks have them in general: sizes that are no power of two, odd
batches, channel counts off the tile sizes, strides, the memory layouts of channels-first and of channels-last
frameworks.  Activations are ReLU outputs, gradients are normal, both drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import torch

from paper_1908_05460_b200 import binding as B
from paper_1908_05460_b200.autograd import GAConv2d
from paper_1908_05460_b200.layers import ConvLayer, layer_set

NETS = {"resnet20": 2, "cnn2": 3, "vgg19": 4}
SCHEDULES = {"every_4th_layer": B.SCHED_EVERY_4TH_LAYER, "alt_layer_alt_batch": B.SCHED_ALT_LAYER_ALT_BATCH,
             "all_layers_every_4th_batch": B.SCHED_ALL_LAYERS_EVERY_4TH_BATCH}
METHODS = {"exact": B.METHOD_EXACT, "zero": B.METHOD_ZERO, "random": B.METHOD_RANDOM, "top1": B.METHOD_TOP1, "topk": B.METHOD_TOPK}
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
# x, dy, dw memory orders: the paper's own; what a channels-first framework holds; what a channels-last one holds
LAYOUTS = {"paper": (B.X_NHWC, B.DY_NKPQ, B.DW_KRSC), "nchw": (B.X_NCHW, B.DY_NKPQ, B.DW_KCRS),
           "nhwc": (B.X_NHWC, B.DY_NPQK, B.DW_KCRS)}


def _layer_case(kind, n, c, h, w, k, r, stride=1, dtype="bf16", layout="paper", **more):
    return dict(kind=kind, n=n, c=c, h=h, w=w, k=k, r=r, stride=stride, dtype=dtype, layout=layout, **more)


def _step_case(net, n, dtype, schedule, method, step, lanes):
    return dict(kind="step", net=net, n=n, dtype=dtype, schedule=schedule, method=method, step=step, lanes=lanes)


def listed():
    def named(name, case):
        return dict(case, name=name)
    return [
        # the smallest call: the benchmark's single-layer configuration, a few images of a narrow fp32 layer
        named("exact_small_f32", _layer_case("exact", 8, 16, 32, 32, 16, 3, dtype="f32")),
        # the middle of VGG-19 at the paper's batch size
        named("exact_vgg_bf16", _layer_case("exact", 128, 256, 8, 8, 256, 3)),
        # the second convolution of the two-layer CNN in fp32, 5x5 filters
        named("exact_cnn_5x5_f32", _layer_case("exact", 128, 64, 16, 16, 64, 5, dtype="f32")),
        # a batch, channel counts and a map that fit no tile, in the layouts a channels-first framework hands over
        named("exact_ragged_bf16", _layer_case("exact", 100, 72, 28, 20, 120, 3, layout="nchw")),
        # a down-sampling layer of a residual network on 28x28 maps, fp32
        named("exact_stride2_f32", _layer_case("exact", 64, 64, 28, 28, 128, 3, stride=2, dtype="f32")),
        # the largest: an early stage of an image network, channels-last gradient as a channels-last framework has it
        named("exact_large_bf16", _layer_case("exact", 64, 128, 56, 56, 128, 3, layout="nhwc")),
        # Algorithm 1 on the layer where it saves most
        named("top1_vgg_bf16", _layer_case("top1", 128, 64, 32, 32, 64, 3)),
        # four entries per map on odd map sizes, fp32, an odd batch
        named("topk_odd_f32", _layer_case("topk", 50, 40, 25, 25, 56, 3, dtype="f32", topk=4)),
        # a layer whose activations and gradients live on the host
        named("host_exact_bf16", _layer_case("host", 128, 64, 16, 16, 128, 3, method="exact")),
        # a training step of the paper's ResNet-20 runs: every fourth layer takes the random gradient
        named("step_resnet20_f32", _step_case("resnet20", 128, "f32", "every_4th_layer", "random", 1, 12)),
        # the schedule sweep's largest step: VGG-19 at batch 256, every fourth layer takes Algorithm 1
        named("step_vgg19_bf16", _step_case("vgg19", 256, "bf16", "every_4th_layer", "top1", 1, 12)),
        # the layer as a training program holds it: forward, input gradient and filter gradient
        named("train_layer_bf16", _layer_case("train", 128, 128, 16, 16, 128, 3, method="exact")),
    ]


# ---- drawn cases ----------------------------------------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo=8, hi=512):
    c = _log(rng, lo, hi)
    t = rng.random()
    return max(8, (c + 8) // 16 * 16) if t < 0.5 else max(8, (c + 4) // 8 * 8) if t < 0.8 else c     # mostly multiples of 16 or 8


def draw(rng):
    big = listed()[5]
    most = work(big)
    while True:
        kind = rng.choice(["exact"] * 5 + ["top1", "topk", "host", "step", "train"])
        if kind == "step":
            return _step_case(rng.choice(sorted(NETS)), _log(rng, 16, 256), rng.choice(["bf16", "f32"]), rng.choice(sorted(SCHEDULES)),
                              rng.choice(["top1", "random", "zero"]), rng.choice([1, 2, 3, 7]), rng.choice([4, 8, 12]))
        n, k = _log(rng, 2, 256), _channels(rng)
        c = 3 if rng.random() < 0.15 else _channels(rng)                                             # image stems
        h = _log(rng, 4, 64)
        w = h if rng.random() < 0.7 else _log(rng, 4, 64)
        r = rng.choice([1, 3, 3, 3, 3, 3, 5, 7]) if min(h, w) >= 8 else rng.choice([1, 3, 3])
        stride = 2 if rng.random() < 0.2 and min(h, w) >= 8 else 1
        more = {"topk": {"topk": rng.choice([2, 3, 4, 8])}, "host": {"method": rng.choice(["exact", "top1"])},
                "train": {"method": rng.choice(["exact", "exact", "top1"])}}.get(kind, {})
        case = _layer_case(kind, n, c, h, w, k, r, stride, rng.choice(["bf16", "bf16", "f32"]),
                           "paper" if kind == "train" else rng.choice(["paper", "paper", "nchw", "nhwc"]), **more)
        wk = work(case)
        if wk["flops"] <= most["flops"] and wk["bytes"] <= (most["bytes"] if kind != "host" else most["bytes"] / 4):
            return case


# ---- inputs and calls -----------------------------------------------------------------------------------------------
def _layer(case):
    return ConvLayer(case["kind"], case["n"], case["c"], case["h"], case["w"], case["k"], case["r"], case["r"], case["stride"],
                     case["r"] // 2)


def _inputs(gen, layer, dtype, x_layout=B.X_NHWC, dy_layout=B.DY_NKPQ):
    """X = max(N(0,1), 0) and dY ~ N(0, 0.01^2) in the memory orders asked for."""
    l = layer
    xs = (l.n, l.h, l.w, l.c) if x_layout == B.X_NHWC else (l.n, l.c, l.h, l.w)
    ds = (l.n, l.k, l.p, l.q) if dy_layout == B.DY_NKPQ else (l.n, l.p, l.q, l.k)
    x = torch.randn(xs, generator=gen, device="cuda").clamp_(min=0.0).to(dtype)
    dy = torch.randn(ds, generator=gen, device="cuda").mul_(l.dy_std).to(dtype)
    return x, dy


def _dw_like(layer, dw_layout, **kw):
    l = layer
    shape = {B.DW_KRSC: (l.k, l.r, l.s, l.c), B.DW_KCRS: (l.k, l.c, l.r, l.s)}[dw_layout]
    return torch.empty(shape, dtype=torch.float32, **kw)


def _sm_budget(layer, elem_bytes):
    """The SM share the benchmark gives a layer of a step: grows with the time its arithmetic or its bytes take."""
    t_us = max(layer.flops_exact() / (1.6e15 if elem_bytes == 2 else 0.8e15), layer.bytes_exact(elem_bytes) / 6.5e12) * 1e6
    return max(18, min(74, int(148 * t_us / 12.0)))


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(190805460 + int(seed))
    dtype = DTYPES[case["dtype"]]
    st = {"kind": case["kind"]}
    if case["kind"] == "step":
        layers = layer_set(NETS[case["net"]], case["n"])
        method = METHODS[case["method"]]
        st["keep"], st["dws"] = [], []
        xs, dys, descs = [], [], []
        for l in layers:
            x, dy = _inputs(gen, l, dtype)
            d = B.make_desc(l, dtype, alpha=1.0 / l.n, sm_budget=_sm_budget(l, x.element_size()))
            st["keep"].append(B.attach_workspace(d))
            xs.append(x); dys.append(dy); descs.append(d)
            st["dws"].append(_dw_like(l, B.DW_KRSC, device="cuda"))
        st["sched"] = B.Schedule(len(layers), SCHEDULES[case["schedule"]], method, 0.0, int(seed))
        st["packed"] = st["sched"].pack_step(xs, dys, st["dws"], descs)
        st["keep"] += xs + dys + descs
        st["step"], st["lanes"] = case["step"], case["lanes"]
        return st
    layer = _layer(case)
    if case["kind"] == "train":
        sched = None if case["method"] == "exact" else B.Schedule(1, B.SCHED_ALL_LAYERS_EVERY_4TH_BATCH, METHODS[case["method"]])
        m = GAConv2d(layer.c, layer.k, layer.r, layer.stride, layer.pad, schedule=sched, dtype=dtype)
        m.step = 3
        with torch.no_grad():
            m.weight.copy_(torch.randn(m.weight.shape, generator=gen, device="cuda") * math.sqrt(2.0 / (layer.c * layer.r * layer.s)))
        x, dy = _inputs(gen, layer, dtype, B.X_NHWC, B.DY_NPQK)
        st["m"], st["x"], st["dy"] = m, x.permute(0, 3, 1, 2).requires_grad_(), dy.permute(0, 3, 1, 2)     # channels-last tensors
        return st
    x_layout, dy_layout, dw_layout = LAYOUTS[case["layout"]]
    st["x"], st["dy"] = _inputs(gen, layer, dtype, x_layout, dy_layout)
    st["dw"] = _dw_like(layer, dw_layout, device="cuda")
    st["desc"] = B.make_desc(layer, dtype, x_layout=x_layout, dy_layout=dy_layout, dw_layout=dw_layout, alpha=1.0 / layer.n,
                             topk=case.get("topk", 1))
    st["method"] = METHODS[case.get("method", case["kind"])]
    st["ws"] = B.attach_workspace(st["desc"], methods=(st["method"],))
    if case["kind"] == "host":
        st["x_host"], st["dy_host"] = st["x"].cpu().pin_memory(), st["dy"].cpu().pin_memory()
        st["dw_host"] = _dw_like(layer, dw_layout).pin_memory()
    return st


def run(st):
    kind = st["kind"]
    if kind == "exact":
        B.gaconv_dw_exact(st["x"], st["dy"], st["dw"], st["desc"])
        return st["dw"]
    if kind in ("top1", "topk"):
        B.gaconv_dw_approx(st["method"], st["x"], st["dy"], st["dw"], st["desc"])
        return st["dw"]
    if kind == "host":
        B.gaconv_dw_from_host(st["method"], st["x_host"], st["dy_host"], st["dw_host"], st["x"], st["dy"], st["dw"], st["desc"])
        return st["dw_host"]
    if kind == "step":
        st["sched"].run_step(st["step"], st["packed"], lanes=st["lanes"])
        return st["dws"]
    y = st["m"](st["x"])
    dx, dw = torch.autograd.grad(y, (st["x"], st["m"].weight), st["dy"])
    return {"y": y.detach(), "dx": dx, "dw": dw}


# ---- what a pass cannot do without, and how closely two correct ones agree ------------------------------------------
def _approx_work(layer, eb, method, topk=1):
    dw = layer.k * layer.c * layer.r * layer.s * 4
    if method in ("zero", "random"):
        return dw, 0
    if method == "exact":
        return layer.bytes_exact(eb), layer.flops_exact()
    patches = topk * layer.n * layer.k * layer.r * layer.s * layer.c
    return layer.n * layer.k * layer.p * layer.q * eb + min(patches, layer.n * layer.c * layer.h * layer.w) * eb + dw, 2 * patches


def _step_methods(case):
    L = len(layer_set(NETS[case["net"]], 1))
    one_based, step = range(1, L + 1), case["step"]
    approx = {"every_4th_layer": [(i - 2) % 4 == 0 and i >= 2 for i in one_based],
              "alt_layer_alt_batch": [i % 2 == 0 and step % 2 == 1 for i in one_based],
              "all_layers_every_4th_batch": [step % 4 == 3] * L}[case["schedule"]]
    return [case["method"] if a else "exact" for a in approx]


def work(case):
    eb = 2 if case["dtype"] == "bf16" else 4
    if case["kind"] == "step":
        parts = [_approx_work(l, eb, m) for l, m in zip(layer_set(NETS[case["net"]], case["n"]), _step_methods(case))]
    else:
        l = _layer(case)
        parts = [_approx_work(l, eb, case.get("method", case["kind"]), case.get("topk", 1))]
        if case["kind"] == "train":      # forward and input gradient on top: W read, Y and dX written, dW in the weight's type
            parts.append(((l.n * l.k * l.p * l.q + l.n * l.c * l.h * l.w + 2 * l.k * l.c * l.r * l.s) * eb - l.k * l.c * l.r * l.s * 4,
                          2 * l.flops_exact()))
    return {"bytes": float(sum(b for b, _ in parts)), "flops": float(sum(f for _, f in parts))}


def tolerance(case):
    """Products and sums are fp32 whatever the inputs' type: orders of summation differ by about 1e-5.  On small maps the
    approximation methods may contract the sparse gradient in the inputs' type, so that a map's sum is rounded to bf16
    once; the module of a bf16 layer returns its results in bf16."""
    if case["kind"] == "train":
        return {"rel": 1e-2} if case["dtype"] == "bf16" else {"rel": 2e-3}       # (fp32 forward and input gradient: the framework's TF32)
    if case["dtype"] == "bf16" and case["kind"] in ("top1", "topk", "host", "step") and case.get("method", "top1") in ("top1", "topk"):
        return {"rel": 4e-3}
    return {"rel": 2e-5}
