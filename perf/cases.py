"""Cases that stand for the work users of this library have it do, each one pass through the public
entry points of `paper_1909_05073_b200.binding`.

Three kinds of pass:
 * "layers": one or several independent packed layers, one `Layer.forward` each, with the workspace
   that a latency-minded caller hands over (`split=True`);
 * "stack": a chain of layers with its max-pools, `Stack.forward` on device buffers or
   `Stack.forward_host` on pinned host buffers;
 * "project": `pconv_project`, dense weights to PCONV weights.

Weights carry both sparsities (4-of-9 patterns, whole kernels removed) and come from
`synth.gen_weights`; activations come from the distributions of the benchmark configurations.
"""
import math
from dataclasses import replace

import torch

from paper_1909_05073_b200 import binding as B
from paper_1909_05073_b200 import synth

PATTERN_SETS = {4: synth.SCP4, 8: synth.PATTERNS8, 12: synth.PATTERNS12}


def _layer(name, c_in, c_out, h, w, n, stride=1, keep=0.3, storage="f32", patterns=8, relu=True, bias=True):
    return dict(name=name, kind="layers", net="single", c_in=c_in, c_out=c_out, h=h, w=w, n=n, stride=stride,
                keep=keep, storage=storage, patterns=patterns, relu=relu, bias=bias)


def _resnet(name, n, storage="f32", keep=0.35):
    return dict(name=name, kind="layers", net="resnet50", n=n, keep=keep, storage=storage, patterns=8, relu=True,
                bias=True)


def _stack(name, size, n, storage="f32", keep=0.3, keep_first=1.0, host=False):
    return dict(name=name, kind="stack", net="vgg16", h=size, w=size, n=n, storage=storage, keep=keep,
                keep_first=keep_first, patterns=8, host=host)


def _project(name, c_out, c_in, keep, patterns=8):
    return dict(name=name, kind="project", c_out=c_out, c_in=c_in, keep=keep, patterns=patterns)


def listed():
    return [
        # the smallest call: one layer, one image (benchmark configuration 1); latency counts
        _layer("layer-64-56x56-n1", 64, 64, 56, 56, 1, keep=0.5),
        # one image through the ImageNet-sized VGG-16 stack: the headline (configuration 2)
        _stack("vgg16-224-n1", 224, 1),
        # the same for a caller whose image and result live on the host
        _stack("vgg16-224-n1-host", 224, 1, host=True),
        # the 3x3 layers of ResNet-50, one image and a served batch (configuration 3)
        _resnet("resnet50-n1", 1),
        _resnet("resnet50-n32", 32),
        # fp16 storage: the CIFAR-sized stack at throughput and at latency (configuration 4)
        _stack("cifar-vgg16-n256-f16", 32, 256, "f16", 0.25, 0.25),
        _stack("cifar-vgg16-n1-f16", 32, 1, "f16", 0.25, 0.25),
        # filters of very different density, stride 1 and 2 (configuration 5)
        _layer("stress-512-14x14-n64", 512, 512, 14, 14, 64, keep=-1.0),
        _layer("stress-512-28x28-s2-n64", 512, 512, 28, 28, 64, stride=2, keep=-1.0),
        # nothing divides anything: ragged channels and maps, the twelve-pattern set, no ReLU, no bias
        _layer("ragged-99-203-45x37-n5-12pat", 99, 203, 45, 37, 5, keep=0.4, patterns=12, relu=False, bias=False),
        # the same for fp16 storage at stride 2
        _layer("ragged-130-75-57x61-s2-n9-f16", 130, 75, 57, 61, 9, stride=2, keep=0.35, storage="f16"),
        # making PCONV weights from dense ones: one training step's projection of a 512-512 layer bank
        _project("project-4096x512", 4096, 512, 0.3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MAX_MACS = 7.0e9     # surviving multiply-adds of a drawn case: below the largest listed one's
MAX_VALUES = 4.0e7   # values of the largest input or output of a drawn case


def draw(rng):
    """One more case of the same ranges: mostly single layers, then stacks, layer sets, projections."""
    u = rng.random()
    if u < 0.1:
        return _plain(_project("", _log_int(rng, 64, 4096), _log_int(rng, 16, 512), rng.uniform(0.1, 0.9),
                               rng.choice([4, 8, 12])))
    while True:
        if u < 0.35:
            c = _stack("", _log_int(rng, 32, 224), _log_int(rng, 1, 256), rng.choice(["f32", "f16"]),
                       rng.uniform(0.2, 0.5), rng.choice([1.0, 0.25]), host=rng.random() < 0.25)
        elif u < 0.45:
            c = _resnet("", _log_int(rng, 1, 32), rng.choice(["f32", "f16"]), rng.uniform(0.25, 0.5))
        else:
            c = _layer("", _log_int(rng, 3, 512), _log_int(rng, 16, 512), _log_int(rng, 7, 224), 0,
                       _log_int(rng, 1, 128), rng.choice([1, 1, 1, 2]),
                       rng.choice([-1.0, rng.uniform(0.2, 0.6), rng.uniform(0.2, 0.6), 1.0]),
                       rng.choice(["f32", "f32", "f16"]), rng.choice([4, 8, 8, 12]), rng.random() < 0.7,
                       rng.random() < 0.7)
            c["w"] = max(7, min(224, int(c["h"] * rng.uniform(0.7, 1.4))))
        values = max(c["n"] * max(s.c_in * s.h * s.w, s.c_out * s.h_out * s.w_out) for s in _specs(c))
        if work(c)["flops"] <= 2 * MAX_MACS and values <= MAX_VALUES:
            return _plain(c)


def _plain(case):
    return {k: v for k, v in case.items() if k != "name"}


def _specs(case):
    """The layer specs of a case."""
    pats = PATTERN_SETS[case["patterns"]]
    probs = (1.0 / len(pats),) * len(pats)
    if case["net"] == "single":
        return [synth.LayerSpec("layer", case["c_in"], case["c_out"], case["h"], case["w"], case["stride"], case["keep"],
                                probs)]
    if case["net"] == "resnet50":
        return [replace(s, keep=case["keep"]) for s in synth.config(3).layers]
    base = synth.config(4 if case["storage"] == "f16" else 2).layers
    out, h = [], case["h"]
    for i, s in enumerate(base):
        out.append(replace(s, h=h, w=h, keep=case["keep_first"] if i == 0 else case["keep"]))
        h = h // 2 if s.pool_after else h
    return out


def _input(spec, n, dtype, gen):
    x = torch.empty((n, spec.c_in, spec.h, spec.w), device="cuda")
    if spec.x_dist == "relu_normal":
        x.normal_(generator=gen).relu_()
    else:
        x.uniform_(0.0 if spec.x_dist == "uniform_01" else -1.0, 1.0, generator=gen)
    return x.to(dtype)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "project":
        w = torch.empty((case["c_out"], case["c_in"], 3, 3), device="cuda")
        return {"w": w.normal_(0.0, 0.05, generator=gen), "patterns": PATTERN_SETS[case["patterns"]],
                "keep": case["keep"], "kind": "project"}
    half = case["storage"] == "f16"
    dtype = torch.float16 if half else torch.float32
    pats = PATTERN_SETS[case["patterns"]]
    specs = _specs(case)
    layers = []
    for i, spec in enumerate(specs):
        w, b, _ = synth.gen_weights(spec, (seed * 64 + i) % (1 << 62), pats)
        layers.append(B.Layer(w, pats, spec.stride, B.F16 if half else B.F32, b if case.get("bias", True) else None,
                              strict4=True))
    n = case["n"]
    state = {"kind": case["kind"], "layers": layers}
    if case["kind"] == "layers":
        state["x"] = [_input(s, n, dtype, gen) for s in specs]
        state["y"] = [torch.empty(l.out_shape(x.shape), dtype=dtype, device="cuda") for l, x in zip(layers, state["x"])]
        state["relu"] = case["relu"]
        return state
    state["stack"] = B.Stack(layers, [s.pool_after for s in specs], n, specs[0].h, specs[0].w, B.RELU)
    x = _input(specs[0], n, dtype, gen)
    y = torch.empty(state["stack"].out_shape, dtype=dtype, device="cuda")
    state["host"] = case["host"]
    if case["host"]:
        x, y = x.cpu().pin_memory(), y.cpu().pin_memory()
        state["stream"] = torch.cuda.Stream()
    state["x"], state["y"] = x, y
    return state


def run(state):
    if state["kind"] == "project":
        return B.pconv_project(state["w"], state["patterns"], state["keep"])
    if state["kind"] == "layers":
        for layer, x, y in zip(state["layers"], state["x"], state["y"]):
            layer.forward(x, relu=state["relu"], out=y, split=True)
        return state["y"]
    if state["host"]:
        state["stack"].forward_host(state["x"], state["y"], state["stream"])
    else:
        state["stack"].forward(state["x"], state["y"])
    return state["y"]


def work(case):
    """Bytes: input, output and bias once, and per surviving kernel its four values and two index
    bytes (a stack's inner activations need not leave the chip).  Operations: two per surviving
    multiply-add; the projection squares nine taps and adds up four of them for every pattern."""
    if case["kind"] == "project":
        n = case["c_out"] * case["c_in"]
        return {"bytes": n * (36 + 36 + 1), "flops": n * (9 + 4 * case["patterns"])}
    es = 2 if case["storage"] == "f16" else 4
    n, specs = case["n"], _specs(case)
    bytes_, flops = 0.0, 0.0
    for i, s in enumerate(specs):
        kept = s.c_in * s.c_out * (0.5 if s.keep < 0 else s.keep)
        flops += 8.0 * kept * n * s.h_out * s.w_out
        bytes_ += kept * (4 * es + 2) + 4 * s.c_out
        if case["kind"] == "layers" or i == 0:
            bytes_ += es * n * s.c_in * s.h * s.w
        if case["kind"] == "layers":
            bytes_ += es * n * s.c_out * s.h_out * s.w_out
        elif i == len(specs) - 1:
            p = 2 if s.pool_after else 1
            bytes_ += es * n * s.c_out * (s.h_out // p) * (s.w_out // p)
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """fp32: sums of up to a few thousand terms in another order.  fp16 storage: one rounding of
    the result per layer (2^-11), which a stack carries through its thirteen layers."""
    if case["kind"] == "project":
        return "exact"
    if case["storage"] == "f16":
        return {"rel": 3e-3 if case["kind"] == "stack" else 1e-3}
    return {"rel": 1e-5}
