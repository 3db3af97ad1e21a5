"""The weight gradient's slices on the pixel grid: more ranges than one pass of the
reduction holds (128), kept filters that are no multiple of its 16-byte loads, dZ
copied in blocks of 1024 slots (the last one ragged), and a layer whose taps are
split between items (longer ranges) at a size where one item could hold them;
against the fp64 oracle, at the suite's 2e-3 of the largest value and, the sums
being fp32 sums of exact products in ranges of at most 6 x 128 pixels, at 2e-6 in
the 2-norm (4.5e-7 measured at most, with 12 x 128)."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from workloads import ConvShape

from _helpers import assert_close

pytestmark = pytest.mark.gpu

CASES = [
    ("ranges_141_filters_18", ConvShape(n=23, c=48, h=28, w=28, f=32, kh=1, kw=1), 18, wl.COL_CHANNEL, 24),
    ("dz_blocks_of_1024", ConvShape(n=32, c=8, h=33, w=33, f=256, kh=1, kw=1), 250, wl.COL_NONE, 0),
    ("split_taps", ConvShape(n=90, c=64, h=14, w=14, f=50, kh=3, kw=3, ph=1, pw=1), 50, wl.COL_NONE, 0),
    ("split_taps_odd_columns", ConvShape(n=90, c=64, h=14, w=14, f=64, kh=3, kw=3, ph=1, pw=1), 61, wl.COL_SHAPE, 301),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c[0])
def test_weight_gradient(case):
    from paper_1807_11091_gb300 import sadmm
    name, s, kf, ck, kc = case
    dev = torch.device("cuda", 0)
    t = wl.gen_tensors(s, seed=3)
    rows, cols, _, _ = oracle.project(t["W"], s.taps, kf, ck, kc)
    fi = torch.as_tensor(rows, dtype=torch.int32, device=dev) if kf < s.f else None
    ci = torch.as_tensor(cols, dtype=torch.int32, device=dev) if ck != wl.COL_NONE else None
    pc = sadmm.PrunedConv(s.desc16(), t["W"].to(dev), fi, ck, ci, kf, kc if ck != wl.COL_NONE else s.k)
    dy = torch.randn(s.y_shape(), generator=torch.Generator().manual_seed(4)).to(torch.bfloat16)
    dW, db, dx = pc.backward(t["x"].to(dev), dy.to(dev), relu=False)
    assert sadmm.device_status() == 0
    rdx, rdW, rdb = oracle.pruned_conv_backward(t["x"], t["W"], t["bias"], s.desc16(), s.taps, rows, ck, cols, dy,
                                                relu=False)
    for got, want, what in ((dW, rdW.reshape(s.f, -1), "dW"), (db, rdb, "db"), (dx, rdx, "dx")):
        g = got.cpu().double().numpy()
        assert_close(g, want, what=f"{name} {what}")
        assert np.linalg.norm(g - want) <= 2e-6 * np.linalg.norm(want), what
    assert np.all(dW.cpu().numpy()[rdW.reshape(s.f, -1) == 0.0] == 0.0)
