"""The pixel-grid backward of a batch whose scratch would pass its bound (256 MiB): the
images in several passes, the last with fewer, dW and db added up over them; against 64
bits, bit for bit the same on every call, and in calls for one of the outputs alone."""
import numpy as np
import pytest
import torch

import workloads as wl
from workloads import ConvShape

pytestmark = pytest.mark.gpu

CASES = [
    # two passes of 13 and 12 images, pruned filters and columns
    ("3x3", ConvShape(n=25, c=64, h=224, w=224, f=64, kh=3, kw=3, ph=1, pw=1), 48, wl.COL_SHAPE, 301),
    # three passes, pruned channels, two conv groups
    ("1x1_groups2", ConvShape(n=37, c=128, h=160, w=160, f=192, kh=1, kw=1, groups=2), 150, wl.COL_CHANNEL, 40),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c[0])
def test_passes_match_64_bits(case):
    from paper_1807_11091_gb300 import sadmm
    name, s, kf, ck, kc = case
    dev = torch.device("cuda", 0)
    g = torch.Generator(device="cuda").manual_seed(15)
    W = torch.randn(s.w_shape(), generator=g, device=dev).to(torch.bfloat16)
    x = torch.relu(torch.randn(s.x_shape(), generator=g, device=dev)).to(torch.bfloat16)
    dy = torch.randn(s.y_shape(), generator=g, device=dev).to(torch.bfloat16)
    y = torch.relu(torch.randn(s.y_shape(), generator=g, device=dev))
    fi, ci, _ = sadmm.project_groups(s.desc16(), W, kf, ck, kc)
    pc = sadmm.PrunedConv(s.desc16(), W, fi, ck, ci, kf, kc)
    # copies of x (the kept channels) and dZ alone, 2 bytes an element, would pass the bound
    copies = 2 * s.n * s.h * s.w * ((s.groups * kc if ck == wl.COL_CHANNEL else s.c) + kf)
    bound = max(256 << 20, sadmm.sadmm_conv_bwd_workspace_size_chunk(pc.plan, 32768))
    assert copies > bound >= sadmm.sadmm_conv_bwd_workspace_size(pc.plan)
    dW, db, dx = pc.backward(x, dy, y=y)
    for want in ((True, True, True), (True, False, False), (False, True, False), (False, False, True)):
        again = pc.backward(x, dy, y=y, want_dw=want[0], want_db=want[1], want_dx=want[2])
        assert all(p is None or torch.equal(p, q) for p, q in zip(again, (dW, db, dx)))
    assert sadmm.device_status() == 0
    keep = torch.zeros(s.f, s.k, dtype=torch.float64, device=dev)
    cols = ci.long() if ck == wl.COL_SHAPE else (ci.long()[:, None] * s.taps + torch.arange(s.taps, device=dev)).reshape(-1)
    keep[fi.long()[:, None], cols[None, :]] = 1.0
    kept = (keep.sum(1) > 0).double()
    Wd = (W.double().reshape(s.f, -1) * keep).reshape(W.shape).requires_grad_(True)
    rW, rb = torch.zeros_like(keep), torch.zeros(s.f, dtype=torch.float64, device=dev)
    err = ref = 0.0
    for n in range(s.n):
        dz = dy[n:n + 1].double() * (y[n:n + 1] > 0) * kept.reshape(1, -1, 1, 1)
        xd = x[n:n + 1].double().requires_grad_(True)
        gx, gw = torch.autograd.grad(torch.nn.functional.conv2d(xd, Wd, padding=(s.ph, s.pw), groups=s.groups), (xd, Wd), dz)
        rW += gw.reshape(s.f, -1) * keep
        rb += dz.sum((0, 2, 3))
        err += (dx[n:n + 1].double() - gx).square().sum().item()
        ref += gx.square().sum().item()
    assert np.sqrt(err / ref) <= 2.5e-7
    assert ((dW.double() - rW).norm() / rW.norm()).item() <= 2.5e-7  # (a pass more adds, rounded, to the ranges' sum)
    assert ((db.double() - rb).norm() / rb.norm()).item() <= 2.5e-7
    assert not dW[keep == 0].any() and not db[kept == 0].any()
