"""What the dense tensor-core kernel makes of values at the ends of the range: largest finite activations
and weights, values so small that a piece of theirs is a bf16 subnormal, and activations that are
infinite or not a number.  The development build pins the kernel, and where it matters its plan
(PCONV_FORCE_DENSE), and the form of its input: NCHW, or position rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_1909_05073_b200 import binding as B
from paper_1909_05073_b200 import build as pbuild
from paper_1909_05073_b200 import synth
from util import check_close

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


def conv_of_surviving_taps(x, wt, bias, stride, relu, storage="f32", pool=False):
    """The layer where infinities and NaNs meet the surviving taps only (no weight inside a pattern is zero
    here): the finite part from the oracle, and from it, on indicator maps, how many terms are infinite."""
    count = lambda hit, w: oracle.conv3x3(hit.astype(np.float32), w.astype(np.float32), None, stride, False) > 0
    with np.errstate(invalid="ignore"):
        up, down, nan = x == np.inf, x == -np.inf, np.isnan(x)
        y = oracle.conv3x3(np.where(np.isfinite(x), x, 0).astype(np.float32), wt, bias, stride, False, storage)
        pos, neg = count(up, wt > 0) | count(down, wt < 0), count(up, wt < 0) | count(down, wt > 0)
        y = np.where(pos, np.inf, np.where(neg, -np.inf, y))
        y = np.where(count(nan, wt != 0) | (pos & neg), np.nan, y).astype(np.float32)
        y = np.fmax(y, 0) if relu else y        # (a maximum with a NaN is the other operand, as on the GPU)
        if pool:
            y = y[:, :, :y.shape[2] // 2 * 2, :y.shape[3] // 2 * 2]
            y = np.fmax(np.fmax(y[:, :, ::2, ::2], y[:, :, ::2, 1::2]), np.fmax(y[:, :, 1::2, ::2], y[:, :, 1::2, 1::2]))
    return y


def check_with_infinities(got, want, storage, what):
    got = got.float().cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want)), "%s: NaN: %d here, %d wanted" % (what, np.isnan(got).sum(), np.isnan(want).sum())
    inf = np.isinf(want)
    assert inf.any() and np.array_equal(got[inf], want[inf]), what
    fine = np.isfinite(want)
    check_close(got[fine], want[fine], storage, what)


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


# The six products of pieces that the dense kernel forms for fp32, each as the only place where a term of
# 2^-18 of the result comes from: 2^-9 is half of a bf16 ulp's half, so 1 + 2^-9 + 2^-18 is cut into these three.
PIECES = [1 + 2.0 ** -9, 1 + 2.0 ** -18 + 2.0 ** -9]


@pytest.mark.parametrize("xv", [1.0] + PIECES)
@pytest.mark.parametrize("wv", [1.0] + PIECES)
def test_no_product_of_pieces_is_left_out(xv, wv, dense):
    """All terms alike: sums of 4 x 20 kept terms of at most 24 bits each.  Leaving x2 w2, x1 w3 or x3 w1 out is an
    error of 3.8e-6 of the result, x1 w2 or x2 w1 one of 2e-3; the products that are left out are below 2^-26
    of it here (x2 w3, x3 w2), and eighty additions in fp32, truncated where the tensor core adds, err by at most
    a twentieth of 2^-18 (measured 1e-7)."""
    c_in, c_out, h, w = 20, 24, 9, 14
    wt = np.zeros((c_out, c_in, 3, 3), np.float32)
    for t in (1, 3, 4, 5):
        wt[:, :, t // 3, t % 3] = wv
    x = np.full((2, c_in, h, w), xv, np.float32)
    layer = B.Layer(wt, synth.PATTERNS8, 1, B.F32, None)
    got = layer.forward(torch.from_numpy(x).cuda(), relu=False).cpu().numpy().astype(np.float64)
    ref = oracle.conv3x3(x, wt, None, 1, False).astype(np.float64)
    assert (np.abs(got - ref) <= 8e-7 * ref).all(), np.abs(got / ref - 1).max()
    layer.close()


@pytest.mark.parametrize("c_in,c_out,h,w,n,stride", [(512, 64, 14, 14, 2, 1), (256, 130, 15, 13, 3, 2), (64, 64, 40, 40, 1, 1)])
def test_fp32_sums_are_as_close_to_64_bits_as_fp32_ones(c_in, c_out, h, w, n, stride, dense):
    """Norm of the error over norm of the result.  A product of pieces left out alone adds 6.5e-7 here; fp32
    sums in any order stay near 1e-7 (the sparse kernel is measured beside it, and allowed the same)."""
    x, wt, bias = make(c_in, c_out, h, w, n, stride)
    layer = B.Layer(wt, synth.PATTERNS8, stride, B.F32, bias)
    xt = torch.from_numpy(x).cuda()
    ref = torch.nn.functional.conv2d(torch.from_numpy(x).double(), torch.from_numpy(wt).double(), torch.from_numpy(bias).double(),
                                     stride, 1).numpy()
    off = {k: np.linalg.norm(layer.forward(xt, relu=False, kernel=k).cpu().numpy() - ref) / np.linalg.norm(ref)
           for k in (0, B.KERNEL_TILED)}
    assert off[B.KERNEL_TILED] <= 3e-7 and off[0] <= 3e-7, off
    layer.close()


SPECIAL = [np.inf, -np.inf, np.nan, np.inf]
CASES = [  # (c_in, c_out, h, w, n, stride): ragged channels and filters, several tiles, strips, parity planes
    (24, 40, 12, 13, 2, 1), (33, 75, 9, 30, 2, 1), (8, 40, 3, 300, 1, 1), (40, 24, 15, 10, 3, 2), (5, 130, 1, 9, 2, 2),
]


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(str(v) for v in c))
def test_infinities_and_nans_reach_only_what_depends_on_them(case, storage, dense):
    c_in, c_out, h, w, n, stride = case
    x, wt, bias = make(c_in, c_out, h, w, n, stride)
    plant(x, SPECIAL, 7)
    layer = B.Layer(wt, synth.PATTERNS8, stride, B.F16 if storage == "f16" else B.F32, bias)
    xt = torch.from_numpy(x).cuda()
    xt = xt.half() if storage == "f16" else xt
    for relu in (False, True):
        for pool in (False, True) if min(layer.out_shape(x.shape)[2:]) > 1 else (False,):
            want = conv_of_surviving_taps(x, wt, bias, stride, relu, storage, pool)
            got = layer.forward(xt, relu=relu, pool=pool)
            check_with_infinities(got, want, storage, "relu=%s pool=%s" % (relu, pool))
    assert B.pconv_device_status(layer.handle) == (0, 0)
    layer.close()


@pytest.mark.parametrize("plan", ["1,64,1,0", "1,64,4,0", "1,64,4,1"])     # whole; parts through the workspace; a cluster
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_infinities_where_thread_blocks_share_a_tile(storage, plan, dense, monkeypatch):
    x, wt, bias = make(256, 64, 7, 7, 1, 1)
    plant(x, SPECIAL, 8)
    monkeypatch.setenv("PCONV_FORCE_DENSE", plan)
    layer = B.Layer(wt, synth.PATTERNS8, 1, B.F16 if storage == "f16" else B.F32, bias)
    xt = torch.from_numpy(x).cuda()
    xt = xt.half() if storage == "f16" else xt
    want = conv_of_surviving_taps(x, wt, bias, 1, False, storage)
    for _ in range(2):                          # the workspace keeps nothing of them
        check_with_infinities(layer.forward(xt, relu=False, split=True), want, storage, plan)
    if layer._ws is not None:
        assert not layer._ws.any()
    layer.close()


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_infinities_through_a_stack(storage, dense):
    """Position rows written by one layer and read by the next, their padding filters among them."""
    chans, pools, strides, h = [17, 40, 24, 72], [1, 0, 0], [1, 2, 1], 21
    x, _, _ = make(17, 8, h, h, 2, 1)
    plant(x, [np.inf, -np.inf], 9)
    layers, a, hh = [], x, h
    for i in range(3):
        _, wt, bias = make(chans[i], chans[i + 1], hh, hh, 1, strides[i], seed=20 + i)
        layers.append(B.Layer(wt, synth.PATTERNS8, strides[i], B.F16 if storage == "f16" else B.F32, bias))
        a = conv_of_surviving_taps(a, wt, bias, strides[i], True, storage, bool(pools[i]))
        if storage == "f16":
            a = a.astype(np.float16).astype(np.float32)
        hh = a.shape[2]
    stack = B.Stack(layers, pools, 2, h, h, B.RELU)
    xt = torch.from_numpy(x).cuda()
    y = torch.empty(stack.out_shape, dtype=torch.float16 if storage == "f16" else torch.float32, device="cuda")
    stack.forward(xt.to(y.dtype), y)
    check_with_infinities(y, a, storage, "stack")
    assert stack.status() == (0, 0)
    stack.close()
