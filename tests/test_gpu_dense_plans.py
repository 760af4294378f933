"""When launch plans of the dense kernel are worked out: planning is host work that a first pass pays for.
The development build counts the plans made."""
import threading
from dataclasses import replace

import pytest
import torch

from paper_1909_05073_b200 import binding as B
from paper_1909_05073_b200 import build as pbuild
from paper_1909_05073_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def dev_library():
    old = B.use_library(pbuild.build(dev=True))
    yield
    B.use_library(None)
    B._lib = old


def made(call):
    """Plans worked out during `call`."""
    before = B.lib().pconv_dev_dense_plans()
    call()
    return B.lib().pconv_dev_dense_plans() - before


def make(c_in, c_out, h, w, n=1, storage="f32", seed=1, stride=1, keep=0.4):
    wt, bias, _ = synth.gen_weights(synth.LayerSpec("p", c_in, c_out, h, w, stride, keep), seed)
    layer = B.Layer(wt, synth.PATTERNS8, stride, B.F16 if storage == "f16" else B.F32, bias)
    x = torch.zeros((n, c_in, h, w), device="cuda")
    return layer, x.half() if storage == "f16" else x


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("flags", [B.KERNEL_TILED, B.KERNEL_SIMPLE, B.KERNEL_GENERIC_TAPS, B.ROWS4, B.ROWS8, B.CLUSTER])
def test_a_pinned_kernel_needs_no_dense_plan(flags, storage):
    layer, x = make(40, 24, 11, 19 + flags.bit_length(), storage=storage)      # (a geometry that no other test has)
    y = torch.empty(layer.out_shape(x.shape), dtype=x.dtype, device="cuda")
    assert made(lambda: B.pconv_forward(layer.handle, x, layer.bias, y, flags | B.RELU)) == 0
    assert made(lambda: B.pconv_forward(layer.handle, x, layer.bias, y, B.RELU)) > 0       # (the choice needs some)
    layer.close()


def test_plans_are_shared_by_layers_of_the_same_geometry_and_by_threads():
    first, x = make(48, 56, 13, 17)
    other, _ = make(48, 56, 13, 17, seed=2)            # other weights, the same geometry
    assert made(lambda: first.forward(x, split=True)) > 0
    assert made(lambda: first.forward(x, split=True)) == 0
    assert made(lambda: other.forward(x, split=True)) == 0
    t = threading.Thread(target=lambda: made_there.append(made(lambda: other.forward(x, split=True))))
    made_there = []
    t.start()
    t.join()
    assert made_there == [0]
    bigger, xb = make(48, 72, 13, 17)                  # another geometry
    assert made(lambda: bigger.forward(xb, split=True)) > 0
    torch.cuda.synchronize()
    for l in (first, other, bigger):
        l.close()


def test_a_workspace_larger_than_needed_changes_no_plan():
    layer, x = make(256, 64, 7, 9)
    need = B.pconv_workspace_bytes(layer.handle, 1, 7, 9)
    assert need > 0
    y = torch.empty(layer.out_shape(x.shape), device="cuda")
    for extra in (0, 256, 1 << 20):
        ws = torch.zeros(need + extra, dtype=torch.uint8, device="cuda")
        assert made(lambda: B.pconv_forward(layer.handle, x, layer.bias, y, B.RELU, workspace=ws)) == 0, extra
        assert not ws.any()
    layer.close()


@pytest.mark.parametrize("case", [
    (512, 512, 14, 14, 64, 1, "f32"), (512, 512, 28, 28, 16, 2, "f32"), (64, 64, 56, 56, 1, 1, "f32"),
    (256, 256, 28, 28, 8, 1, "f32"), (130, 75, 57, 61, 9, 2, "f16"), (256, 256, 56, 56, 1, 1, "f32"),
    (64, 64, 32, 32, 64, 1, "f16"), (512, 512, 4, 4, 64, 1, "f16"), (33, 60, 19, 23, 3, 1, "f16"),
], ids=lambda c: "x".join(str(v) for v in c))
def test_scratch_is_asked_for_where_a_forward_uses_it_and_nowhere_else(case):
    c_in, c_out, h, w, n, stride, storage = case
    layer, x = make(c_in, c_out, h, w, n, storage, 3, stride)
    x.uniform_(0.5, 1.5)
    need = B.pconv_scratch_bytes(layer.handle, n, h, w)
    ws = layer.workspace(x.shape)
    touched = 0
    for pool in (False, True) if stride == 1 else (False,):
        for workspace in {id(ws): ws, id(None): None}.values():
            room = torch.full((256 << 20,), 0xA5, dtype=torch.uint8, device="cuda")
            _, co, ho, wo = layer.out_shape(x.shape)
            y = torch.empty((n, co, ho // 2, wo // 2) if pool else (n, co, ho, wo), dtype=x.dtype, device="cuda")
            B.pconv_forward(layer.handle, x, layer.bias, y, B.RELU | (B.POOL2X2 if pool else 0), workspace=workspace, scratch=room)
            used = (room != 0xA5).nonzero()
            touched = max(touched, int(used.max()) + 1 if len(used) else 0)
    assert touched <= need, "a forward used more than was asked for"
    assert (touched > 0) == (need > 0), "%d bytes asked for, %d used" % (need, touched)
    assert B.pconv_device_status(layer.handle) == (0, 0)
    layer.close()


def test_a_first_forward_plans_only_what_it_may_run():
    """The sizes of workspace and scratch, which are asked for before it, need NCHW plans (plain and pooled, with
    a workspace and without) and one on position rows for each where staging them could pay; nothing is left
    for the forward itself, nor where its result is pooled."""
    for c, h, w, most in ((64, 54, 47, 8), (256, 15, 13, 8), (3, 9, 20, 4)):
        layer, x = make(c, c, h, w)
        sizes = made(lambda: (layer.workspace(x.shape), layer.scratch(x.shape)))
        assert 0 < sizes <= most, (c, h, w, sizes)
        for pool in (False, True):
            assert made(lambda: layer.forward(x, split=True, pool=pool)) == 0, (c, h, w)
            assert made(lambda: layer.forward(x, pool=pool)) == 0, (c, h, w)
        layer.close()


def test_a_stack_with_a_pinned_kernel_plans_nothing():
    layers = [make(24, 40, 23, 21)[0], make(40, 16, 23, 21)[0]]
    for flags in (B.KERNEL_TILED, B.KERNEL_SIMPLE, B.ROWS4):
        assert made(lambda: B.Stack(layers, [False, True], 1, 23, 21, B.RELU | flags)) == 0
    assert made(lambda: B.Stack(layers, [False, True], 1, 23, 21, B.RELU)) > 0
    for l in layers:
        l.close()


SPARSE, NCHW, ROWS = 0, 1, 2
ROOM, GIVEN = 1, 2
MEASURED = [  # c_in, c_out, h, w, n, stride, keep, storage, rows, the fastest, and what was measured (us)
    (256, 256, 28, 28, 2, 1, 0.3, "f32", GIVEN, SPARSE),     # 24.0; on rows 32.6
    (256, 256, 12, 12, 8, 1, 0.3, "f32", GIVEN, SPARSE),     # 22.6; on rows 32.2
    (512, 512, 16, 16, 1, 1, 0.3, "f32", GIVEN, SPARSE),     # 18.0; on rows 22.7
    (512, 512, 28, 28, 1, 1, 0.3, "f32", GIVEN, ROWS),       # 32.2; sparse 39.9
    (512, 512, 20, 20, 4, 1, 0.3, "f32", GIVEN, ROWS),       # 66.3; sparse 89.8
    (512, 512, 14, 14, 64, 1, 0.5, "f32", ROOM, NCHW),       # 310; sparse 589
    (512, 512, 7, 7, 1, 1, 0.3, "f16", GIVEN, ROWS),         # 8.4; sparse 23.8
]


@pytest.mark.parametrize("case", MEASURED, ids=lambda c: "x".join(str(v) for v in c))
def test_the_choice_of_kernel_where_measurements_are_far_apart(case):
    c_in, c_out, h, w, n, stride, keep, storage, rows, fastest = case
    layer, _ = make(c_in, c_out, 9, 9, 1, storage, 2, stride, keep)
    ws = B.pconv_workspace_bytes(layer.handle, n, h, w)
    for _ in range(2):                              # (worked out, then found)
        assert B.lib().pconv_dev_path(layer.handle, n, h, w, 0, rows, ws) == fastest
    layer.close()


@pytest.mark.parametrize("size,n,keep,sparse", [(64, 4, 0.3, True), (64, 8, 0.3, True), (224, 1, 0.3, False), (64, 4, 0.5, False)])
def test_a_stack_that_runs_faster_on_the_sparse_kernel_throughout_does_so(size, n, keep, sparse):
    """VGG-16, measured: 236 us as chosen layer by layer against 216 sparse, 299 against 272, 350 against 369, 238
    against 252."""
    layers, pools, h = [], [], size
    for i, s in enumerate(synth.config(2).layers):
        wt, b, _ = synth.gen_weights(replace(s, keep=1.0 if i == 0 else keep, h=h, w=h), 7 + i)
        layers.append(B.Layer(wt, synth.PATTERNS8, 1, B.F32, b))
        pools.append(s.pool_after)
        h = h // 2 if s.pool_after else h
    stack = B.Stack(layers, pools, n, size, size, B.RELU)
    pinned = B.Stack(layers, pools, n, size, size, B.RELU | B.KERNEL_TILED)
    assert (B.lib().pconv_dev_stack_dense_layers(stack.ptr) == 0) == sparse
    assert stack.launches() == len(layers)
    x = torch.rand((n, 3, size, size), device="cuda")
    y, z = torch.empty(stack.out_shape, device="cuda"), torch.empty(stack.out_shape, device="cuda")
    for _ in range(2):
        stack.forward(x, y)
        pinned.forward(x, z)
    assert float((y - z).norm() / z.norm()) < 1e-5          # sums of up to 4608 terms in another order, thirteen times
    assert stack.status() == (0, 0) and pinned.status() == (0, 0)
    stack.close()
    pinned.close()
