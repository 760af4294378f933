"""When launch plans of the dense kernel are worked out: planning is host work that a first pass pays for.
The development build counts the plans made."""
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


def make(c_in, c_out, h, w, n=1, storage="f32", seed=1, stride=1):
    wt, bias, _ = synth.gen_weights(synth.LayerSpec("p", c_in, c_out, h, w, stride, 0.4), seed)
    layer = B.Layer(wt, synth.PATTERNS8, stride, B.F16 if storage == "f16" else B.F32, bias)
    x = torch.zeros((n, c_in, h, w), device="cuda")
    return layer, x.half() if storage == "f16" else x


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("flags", [B.KERNEL_TILED, B.KERNEL_SIMPLE, B.KERNEL_GENERIC_TAPS, B.ROWS4, B.ROWS8, B.CLUSTER])
def test_a_pinned_kernel_needs_no_dense_plan(flags, storage):
    layer, x = make(40, 24, 11, 19, storage=storage)
    y = torch.empty(layer.out_shape(x.shape), dtype=x.dtype, device="cuda")
    assert made(lambda: B.pconv_forward(layer.handle, x, layer.bias, y, flags | B.RELU)) == 0
    assert made(lambda: B.pconv_forward(layer.handle, x, layer.bias, y, B.RELU)) > 0       # (the choice needs some)
    layer.close()
