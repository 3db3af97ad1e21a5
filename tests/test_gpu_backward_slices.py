"""The weight gradient on the pixel grid: its slices (kept filters that are no multiple of
the reduction's 16-byte loads, several pixel ranges), dZ copied in blocks of 1024 slots
(the last one ragged), a layer whose taps are split between items, and groups that keep
more filters than an item's taps were set for; against the fp64 oracle, at the suite's
2e-3 of the largest value and, the sums being fp32 sums of exact products, at 2e-6 in the
2-norm, or at the bound that a test derives."""
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


@pytest.mark.parametrize("case", [
    ("3x3", ConvShape(n=24, c=64, h=56, w=56, f=64, kh=3, kw=3, ph=1, pw=1)),  # ranges of the most tiles
    ("1x1", ConvShape(n=16, c=256, h=28, w=28, f=160, kh=1, kw=1)),
    ("13x13", ConvShape(n=128, c=256, h=13, w=13, f=96, kh=3, kw=3, ph=1, pw=1)),  # two channel blocks
    ("wide", ConvShape(n=8, c=144, h=14, w=14, f=520, kh=3, kw=3, ph=1, pw=1)),  # filter tiles below 256
], ids=lambda c: c[0])
def test_weight_gradient_error_against_64_bits(case):
    """dW in the 2-norm against 64 bits: the tensor core truncates about 5e-9 of a sum per step
    of 16 pixels and its sums are 16 steps long, which the at most 32 fp32 additions of a range
    and those of the ranges raise to 1.6e-7.  Sums of 48 steps stand at 2.0 to 2.7e-7."""
    from paper_1807_11091_gb300 import sadmm
    name, s = case
    dev = torch.device("cuda", 0)
    g = torch.Generator().manual_seed(12)
    W = torch.randn(s.w_shape(), generator=g).to(torch.bfloat16).to(dev)
    x = torch.relu(torch.randn(s.x_shape(), generator=g)).to(torch.bfloat16).to(dev)
    dy = torch.randn(s.y_shape(), generator=g).to(torch.bfloat16).to(dev)
    pc = sadmm.PrunedConv(s.desc16(), W, None, wl.COL_NONE, None, s.f, s.k)
    dW = pc.backward(x, dy, relu=False, want_dx=False)[0]
    assert sadmm.device_status() == 0
    ref = _dw64(s, x, dy)
    assert ((dW.double().reshape(s.f, -1) - ref).norm() / ref.norm()).item() <= 1.8e-7


def _dw64(s, x, dy):
    Wd = torch.zeros(s.w_shape(), dtype=torch.float64, device=x.device, requires_grad=True)
    y = torch.nn.functional.conv2d(x.double(), Wd, padding=(s.ph, s.pw), groups=s.groups)
    return torch.autograd.grad(y, Wd, dy.double())[0].reshape(s.f, -1)


@pytest.mark.parametrize("kept", [(128, 2), (3, 128), (128, 0), (64, 66)], ids=str)
def test_weight_gradient_of_uneven_groups(kept):
    """The taps of an item are set for the filters a group is likely to keep; a group that keeps
    more takes several passes over the pixels, one that keeps none has no items."""
    from paper_1807_11091_gb300 import sadmm
    s = ConvShape(n=6, c=48, h=15, w=14, f=256, kh=5, kw=5, ph=2, pw=2, groups=2)
    dev = torch.device("cuda", 0)
    g = torch.Generator().manual_seed(13)
    W = torch.randn(s.w_shape(), generator=g).to(torch.bfloat16).to(dev)
    x = torch.relu(torch.randn(s.x_shape(), generator=g)).to(torch.bfloat16).to(dev)
    dy = torch.randn(s.y_shape(), generator=g).to(torch.bfloat16).to(dev)
    rows = np.concatenate([np.arange(kept[0]), 128 + np.arange(kept[1])]).astype(np.int32)
    pc = sadmm.PrunedConv(s.desc16(), W, torch.as_tensor(rows, device=dev), wl.COL_NONE, None, len(rows), s.k)
    dW, _, dx = pc.backward(x, dy, relu=False)
    assert sadmm.device_status() == 0
    ref = _dw64(s, x, dy)
    keep = torch.zeros(s.f, 1, dtype=torch.float64, device=dev)
    keep[torch.as_tensor(rows, device=dev).long()] = 1.0
    ref = ref * keep
    assert ((dW.double().reshape(s.f, -1) - ref).norm() / ref.norm()).item() <= 1.8e-7
    assert not dW.reshape(s.f, -1)[keep[:, 0] == 0].any()
    xd = x.double().requires_grad_(True)
    Wd = (W.double().reshape(s.f, -1) * keep).reshape(W.shape)
    rdx, = torch.autograd.grad(torch.nn.functional.conv2d(xd, Wd, padding=(2, 2), groups=2), xd, dy.double())
    assert ((dx.double() - rdx).norm() / rdx.norm()).item() <= 2.5e-7


@pytest.mark.parametrize("n,c,f,hw,kc", [
    (1, 256, 300, 7, 2301), (1, 128, 300, 7, 1151), (1, 64, 300, 7, 570), (8, 40, 100, 14, 353), (4, 16, 20, 9, 143),
    (64, 64, 64, 28, 301), (128, 256, 96, 13, 577),
], ids=lambda v: str(v))
def test_slice_reduction_by_ranges_and_blocks(n, c, f, hw, kc):
    """The reduction's range lanes follow the ranges (one range of a wide layer to 47 of a
    narrow one) and its blocks; columns and filters that are no multiple of a block's."""
    from paper_1807_11091_gb300 import sadmm
    s = ConvShape(n=n, c=c, h=hw, w=hw, f=f, kh=3, kw=3, ph=1, pw=1)
    dev = torch.device("cuda", 0)
    g = torch.Generator().manual_seed(14)
    W = torch.randn(s.w_shape(), generator=g).to(torch.bfloat16).to(dev)
    x = torch.relu(torch.randn(s.x_shape(), generator=g)).to(torch.bfloat16).to(dev)
    dy = torch.randn(s.y_shape(), generator=g).to(torch.bfloat16).to(dev)
    rows, cols = np.sort(np.random.default_rng(1).permutation(f)[:f - 3]), np.sort(np.random.default_rng(2).permutation(s.k)[:kc])
    fi, ci = (torch.as_tensor(a.astype(np.int32), device=dev) for a in (rows, cols))
    pc = sadmm.PrunedConv(s.desc16(), W, fi, wl.COL_SHAPE, ci, f - 3, kc)
    dW, db, _ = pc.backward(x, dy, relu=False)
    assert sadmm.device_status() == 0
    keep = torch.zeros(f, s.k, dtype=torch.float64, device=dev)
    keep[fi.long()[:, None], ci.long()[None, :]] = 1.0
    ref = _dw64(s, x, dy) * keep
    dW = dW.double().reshape(f, -1)
    assert ((dW - ref).norm() / ref.norm()).item() <= 1.8e-7
    assert not dW[keep == 0].any()
    rdb = dy.double().sum((0, 2, 3)) * (keep.sum(1) > 0)
    assert (db.double() - rdb).abs().max().item() <= 1e-5 * rdb.abs().max().item()
