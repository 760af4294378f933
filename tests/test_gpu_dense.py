"""GPU parity of the dense tensor-core kernel for both storage types, where it can go wrong: tiles of 128
positions and up to 128 filters that are just missed or just passed, channel counts around a step of
16, maps of one pixel and of one row, column strips, both strides, the fused pool, tap sets smaller than
nine, tiles shared by several thread blocks, and both forms of the input (NCHW and position rows).  The
development build pins the kernel and the form; the layers' own choice is tried beside them."""
import numpy as np
import pytest
import torch

import oracle
from paper_1909_05073_b200 import binding as B
from paper_1909_05073_b200 import build as pbuild
from paper_1909_05073_b200 import synth
from util import Guarded, check_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def dev_library():
    old = B.use_library(pbuild.build(dev=True))
    yield
    B.use_library(None)
    B._lib = old


CASES = [  # (c_in, c_out, h, w, n, stride, patterns)
    (1, 1, 1, 1, 1, 1, synth.PATTERNS8),
    (15, 16, 1, 127, 1, 1, synth.PATTERNS8),      # one row; positions just below / at / above a tile
    (16, 17, 7, 15, 1, 1, synth.PATTERNS8),
    (17, 15, 3, 42, 1, 1, synth.PATTERNS8),
    (33, 127, 9, 13, 2, 1, synth.SCP4),           # five taps only
    (32, 129, 14, 14, 2, 1, synth.PATTERNS8),     # two filter tiles, the second nearly empty
    (48, 208, 5, 5, 9, 1, synth.PATTERNS12),
    (20, 260, 8, 8, 20, 1, synth.PATTERNS8),
    (8, 40, 3, 300, 1, 1, synth.PATTERNS8),       # wider than a column strip
    (64, 64, 28, 28, 1, 2, synth.PATTERNS8),
    (24, 100, 9, 11, 3, 2, synth.PATTERNS12),
    (130, 75, 1, 9, 2, 2, synth.PATTERNS8),
    (256, 128, 7, 7, 1, 1, synth.PATTERNS8),      # few tiles, many steps: tiles shared by thread blocks
    (512, 96, 4, 6, 2, 1, synth.PATTERNS8),
]


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(str(v) for v in c[:6]))
def test_dense_kernel_matches_the_oracle_from_both_forms_of_the_input(case, storage, monkeypatch):
    c_in, c_out, h, w, n, stride, pats = case
    # (a layer without any kernel has no dense weights: the smallest one keeps its only kernel)
    spec = synth.LayerSpec("t", c_in, c_out, h, w, stride, 1.0 if c_in * c_out == 1 else 0.7, (1.0 / len(pats),) * len(pats))
    wt, bias, _ = synth.gen_weights(spec, 300 + c_in + c_out, pats)
    x = synth.gen_input(spec, n, 300 + c_in)
    layer = B.Layer(wt, pats, stride, B.F16 if storage == "f16" else B.F32, bias)
    xt = torch.from_numpy(x).cuda()
    xt = xt.half() if storage == "f16" else xt
    ref = oracle.conv3x3(x, wt, bias, stride, True, storage)
    pooled = [False] + ([True] if min(ref.shape[2:]) >= 2 else [])
    for pool in pooled:
        want = oracle.maxpool2x2(ref) if pool else ref
        for split in (False, True):
            ws = layer.workspace(xt.shape) if split else None
            for form in ("chosen", "nchw", "rows"):
                with monkeypatch.context() as m:
                    if form != "chosen":
                        m.setenv("PCONV_FORCE_DENSE", "0,0,0,0")
                        m.setenv("PCONV_FORCE_ROWS", "1" if form == "rows" else "0")
                    need = B.pconv_scratch_bytes(layer.handle, n, h, w)
                    assert need > 0 if form == "rows" else need == 0 or form == "chosen"
                    scratch = Guarded((need,), torch.uint8, fill=0xFF) if need else None     # (NaNs, where nothing is staged)
                    y = Guarded(want.shape, xt.dtype, fill=float("nan"))
                    B.pconv_forward(layer.handle, xt, layer.bias, y.t, B.RELU | (B.POOL2X2 if pool else 0), workspace=ws,
                                    scratch=scratch and scratch.t)
                    y.check("output")
                    if scratch:
                        scratch.check("scratch")
                        # (stride 2 with a pool has no dense form: the tiled kernel runs)
                        assert form != "rows" or (pool and stride == 2) or (scratch.t != 0xFF).any()
                check_close(y.t.float().cpu().numpy(), want, storage, "pool=%s split=%s %s" % (pool, split, form))
        if layer._ws is not None:
            assert not layer._ws.any()
    assert B.pconv_device_status(layer.handle) == (0, 0)
    layer.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("n,h,w", [(1, 32, 32), (3, 37, 29), (40, 8, 8)])
def test_stack_that_hands_position_rows_from_layer_to_layer(n, h, w, storage, monkeypatch):
    """Layers of ragged widths, pools and a stride-2 layer: every kind of row layout is written by one
    layer and read by the next (the dense kernel on rows pinned: six launches, one of which stages)."""
    monkeypatch.setenv("PCONV_FORCE_DENSE", "0,0,0,0")
    monkeypatch.setenv("PCONV_FORCE_ROWS", "1")
    chans, pools, strides = [17, 40, 100, 256, 260, 20], [0, 1, 0, 0, 1], [1, 1, 2, 1, 1]
    dt = torch.float16 if storage == "f16" else torch.float32
    specs = [synth.LayerSpec("l%d" % i, chans[i], chans[i + 1], h, w, strides[i], 0.4, sigma=None) for i in range(5)]
    x = synth.gen_input(specs[0], n, 11)
    a, layers = x, []
    for i, s in enumerate(specs):
        wt, b, _ = synth.gen_weights(s, 40 + i)
        layers.append(B.Layer(wt, synth.PATTERNS8, strides[i], B.F16 if storage == "f16" else B.F32, b))
        a = oracle.conv3x3(a, wt, b, strides[i], True, storage)
        if storage == "f16":
            a = a.astype(np.float16).astype(np.float32)
        a = oracle.maxpool2x2(a) if pools[i] else a
    stack = B.Stack(layers, pools, n, h, w, B.RELU)
    assert stack.launches() == 6
    y = Guarded(stack.out_shape, dt, fill=float("nan"))
    for _ in range(2):
        stack.forward(torch.from_numpy(x).cuda().to(dt), y.t)
        y.check("stack output")
        check_close(y.t.float().cpu().numpy(), a, storage, "stack")
    assert stack.status() == (0, 0)
    stack.close()
