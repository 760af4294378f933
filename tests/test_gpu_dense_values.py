"""What the dense tensor-core kernel makes of values at the ends of the fp32 range: largest finite
activations and weights, and values so small that a piece of theirs is a bf16 subnormal.  The development
build pins the kernel (PCONV_FORCE_DENSE) and the form of its input: NCHW, or position rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_1909_05073_b200 import binding as B
from paper_1909_05073_b200 import build as pbuild
from paper_1909_05073_b200 import synth

pytestmark = pytest.mark.gpu

FLT_MAX = float(np.finfo(np.float32).max)


@pytest.fixture(scope="module", autouse=True)
def dev_library():
    old = B.use_library(pbuild.build(dev=True))
    yield
    B.use_library(None)
    B._lib = old


@pytest.fixture(params=["nchw", "rows"])
def dense(request, monkeypatch):
    monkeypatch.setenv("PCONV_FORCE_DENSE", "0,0,0,0")
    monkeypatch.setenv("PCONV_FORCE_ROWS", "1" if request.param == "rows" else "0")


def make(c_in, c_out, h, w, n, stride, storage="f32", seed=5, keep=0.5):
    spec = synth.LayerSpec("v", c_in, c_out, h, w, stride, keep)
    wt, bias, _ = synth.gen_weights(spec, seed)
    x = np.random.default_rng(seed).uniform(-1, 1, (n, c_in, h, w)).astype(np.float32)
    return x, wt, bias


def plant(a, values, seed):
    """`values` at random places of the non-zero entries of `a`."""
    at = np.random.default_rng(seed).choice(np.flatnonzero(a), len(values), replace=False)
    a.ravel()[at] = np.asarray(values, np.float32)


# 0x7F7F8000 is the smallest magnitude that bf16 rounds to infinity
ENDS = [FLT_MAX, -FLT_MAX] + [s * float(np.uint32(b).view(np.float32)) for s in (1, -1) for b in (0x7F7F8000, 0x7F7F7FFF)]
TINY = [2.0 ** -110, -3e-37, 1.1754944e-38, 1e-40, -1e-45]


@pytest.mark.parametrize("where", ["x", "w"])
@pytest.mark.parametrize("c_in,c_out,h,w,n,stride", [(24, 40, 12, 13, 2, 1), (40, 24, 15, 10, 1, 2), (64, 16, 5, 6, 1, 1)])
def test_largest_and_smallest_finite_values(c_in, c_out, h, w, n, stride, where, dense):
    x, wt, bias = make(c_in, c_out, h, w, n, stride)
    if where == "x":
        wt *= np.float32(0.1)                   # (no sum leaves the range)
        plant(x, ENDS + TINY, 6)
    else:
        x *= np.float32(1e-3)
        plant(wt, ENDS + TINY, 6)
    layer = B.Layer(wt, synth.PATTERNS8, stride, B.F32, bias)
    got = layer.forward(torch.from_numpy(x).cuda(), relu=False).cpu().numpy().astype(np.float64)
    assert B.pconv_device_status(layer.handle) == (0, 0)
    ref = oracle.conv3x3(x, wt, bias, stride, False).astype(np.float64)
    # products that are left out and fp32 sums of 4 c_in terms, in the order and with the truncation of the
    # tensor core: each at most 2^-23 of the sum of the terms' magnitudes
    size = oracle.conv3x3(np.abs(x), np.abs(wt), np.abs(bias), stride, False).astype(np.float64)
    assert np.isfinite(size).all()
    assert np.isfinite(got).all(), "%d outputs are not finite" % (~np.isfinite(got)).sum()
    assert (np.abs(got - ref) <= (4 * c_in + 8) * 2.0 ** -23 * size).all()
    layer.close()
