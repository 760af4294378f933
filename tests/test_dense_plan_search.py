"""The dense kernel's launch plans as host arithmetic, through the development build: the search that leaves
candidates out finds the plan that the search through all of them finds, and a plan fits the hardware and
the caller's workspace."""
import ctypes

import numpy as np
import pytest

from paper_1909_05073_b200 import binding as B
from paper_1909_05073_b200 import build as pbuild

FIELDS = ("tiles", "nt", "grid", "split", "cluster", "parts", "n_tiles", "k_steps", "a_stages", "b_slots", "smem",
          "columns", "need", "share")


@pytest.fixture(scope="module")
def lib():
    return B.load(pbuild.build(dev=True))


def plan(lib, shape, ws, clusters, prune):
    out, cycles = (ctypes.c_int * len(FIELDS))(), ctypes.c_double(0)
    st = lib.pconv_dev_dense_plan(*shape, ws, clusters, prune, out, ctypes.byref(cycles))
    return (dict(zip(FIELDS, out)), cycles.value) if st == B.OK else None


def test_pruned_search_finds_the_same_plan_and_plans_fit(lib):
    rng = np.random.default_rng(31)
    pick = lambda *v: int(v[rng.integers(len(v))])
    found = kinds = 0
    for _ in range(1500):
        c_out, c_in = pick(1, 16, 40, 64, 75, 128, 203, 256, 512, 1000), pick(1, 3, 16, 40, 64, 99, 256, 512, 1024)
        h, w, n = pick(1, 2, 7, 14, 28, 45, 56, 112, 224), pick(1, 2, 3, 7, 14, 28, 37, 56, 112, 300), pick(1, 1, 2, 9, 32, 256)
        stride, storage, taps = pick(1, 1, 2), pick(B.F32, B.F16), pick(0x1FF, 0x0BA, 0x01B)
        pool = pick(0, 1) if stride == 1 and min(h, w) > 1 else 0
        shape = (c_out, c_in, stride, storage, taps, n, h, w, pool, pick(0, 1))
        ws, clusters = pick(0, 1 << 17, 1 << 21, 24 << 20), pick(0, 100, 148)
        p = plan(lib, shape, ws, clusters, 1)
        assert p == plan(lib, shape, ws, clusters, 0), (shape, ws, clusters)
        if p is None:
            continue
        found += 1
        g, _ = p
        what = (shape, ws, clusters, g)
        assert g["smem"] <= 227 * 1024 and 1 <= g["a_stages"] <= 4 and g["b_slots"] <= 24, what
        assert g["columns"] <= 512 and g["nt"] % 16 == 0 and g["nt"] <= 128, what
        assert 1 <= g["grid"] <= 148 and g["need"] <= ws, what
        if g["cluster"]:
            assert 2 <= g["parts"] <= 8 and g["n_tiles"] <= clusters // g["parts"] and g["need"] == 0, what
        kinds |= 1 << (2 * g["split"] + g["cluster"])
        # a workspace between what the plan needs and what it was made for gives the same plan
        for less in {g["need"], (g["need"] + ws) // 2}:
            assert plan(lib, shape, less, clusters, 1) == p, (what, less)
    assert found > 1000 and kinds == 0b1101, (found, kinds)
