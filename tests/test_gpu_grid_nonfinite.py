"""Non-finite values on the pixel grid's paths.  A zero of the padded copies that met one
makes a NaN the kept terms do not have, so an entry that comes out NaN is summed again: no
further than its first NaN term, and of a weight gradient only the pixel ranges that came
out NaN.  A diverged training step (NaN everywhere) must not take many times a finite one,
and a sum taken again is as exact as the others."""
import numpy as np
import pytest
import torch

import workloads as wl
from workloads import ConvShape

pytestmark = pytest.mark.gpu

S = ConvShape(n=64, c=96, h=27, w=27, f=256, kh=5, kw=5, ph=2, pw=2, groups=2)


def _layer(s, kf, kc):
    from paper_1807_11091_gb300 import sadmm
    dev = torch.device("cuda", 0)
    g = torch.Generator(device="cuda").manual_seed(16)
    W = torch.randn(s.w_shape(), generator=g, device=dev).to(torch.bfloat16)
    x = torch.relu(torch.randn(s.x_shape(), generator=g, device=dev)).to(torch.bfloat16)
    dy = torch.randn(s.y_shape(), generator=g, device=dev).to(torch.bfloat16)
    fi, ci, _ = sadmm.project_groups(s.desc16(), W, kf, wl.COL_SHAPE, kc)
    pc = sadmm.PrunedConv(s.desc16(), W, fi, wl.COL_SHAPE, ci, kf, kc)
    keep = torch.zeros(s.f, s.k, dtype=torch.bool, device=dev)
    keep[fi.long()[:, None], ci.long()[None, :]] = True
    return pc, W, x, dy, keep


def _us(call):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(2):
        call()
    a.record()
    for _ in range(3):
        call()
    b.record()
    b.synchronize()
    return a.elapsed_time(b) * 1000 / 3


@pytest.mark.parametrize("what", ["dy", "x", "dy_filter", "dy_pixel"])
def test_nan_backward(what):
    from paper_1807_11091_gb300 import sadmm
    pc, W, x, dy, keep = _layer(S, 128, 600)
    f0 = int(torch.nonzero(keep.any(1))[-1])
    xn, dyn = x.clone(), dy.clone()
    if what == "dy":
        dyn.fill_(float("nan"))
    elif what == "x":
        xn.fill_(float("nan"))
    elif what == "dy_filter":
        dyn[:, f0] = float("nan")
    else:
        dyn[S.n - 1, f0, 20, 20] = float("nan")
    clean = _us(lambda: pc.backward(x, dy, relu=False))
    bad = _us(lambda: pc.backward(xn, dyn, relu=False))
    dW, db, dx = pc.backward(xn, dyn, relu=False)
    want = keep.clone()
    if what.startswith("dy_"):
        want[torch.arange(S.f, device=dW.device) != f0] = False
    assert torch.equal(torch.isnan(dW.reshape(S.f, -1)), want) and sadmm.device_status() == 0
    # (one NaN filter or pixel: the NaN term of an output is not among the first that are looked at)
    assert bad <= {"x": 20, "dy": 40}.get(what, 60) * clean, (bad, clean)


def test_nan_forward():
    pc, W, x, dy, keep = _layer(S, 128, 600)
    assert pc.plan.gx_mode == 1
    clean = _us(lambda: pc.forward(x, None, relu=False))
    xn = torch.full_like(x, float("nan"))
    bad = _us(lambda: pc.forward(xn, None, relu=False))
    y = pc.forward(xn, None, relu=False)
    assert torch.equal(torch.isnan(y).flatten(2).all(2), keep.any(1)[None].expand(S.n, -1))
    assert bad <= 20 * clean, (bad, clean)


def test_sums_taken_again_are_exact():
    """One infinity in x at an image's corner: the weight gradient of every tap of its channel
    comes out NaN first, that of the taps that do not read the pixel is finite after all; in
    the forward, that of the outputs whose tap on it is pruned."""
    from paper_1807_11091_gb300 import sadmm
    s = ConvShape(n=128, c=48, h=28, w=28, f=96, kh=3, kw=3, ph=1, pw=1)
    pc, W, x, dy, keep = _layer(s, 96, 400)
    assert s.m > 100000
    c0 = int(keep[0].reshape(s.c, 9).sum(1).float().argmax())
    xi = x.clone()
    xi[70, c0, 0, 0] = float("inf")
    dW, _, _ = pc.backward(xi, dy, relu=False)
    bad = ~torch.isfinite(dW.reshape(s.f, s.c, 3, 3))
    k4 = keep.reshape(s.f, s.c, 3, 3)
    seen = torch.zeros_like(bad)
    seen[:, c0, :2, :2] = True  # read by output (1 - kh, 1 - kw)
    assert torch.equal(bad, seen & k4)
    Wd = torch.zeros(s.w_shape(), dtype=torch.float64, device=x.device, requires_grad=True)
    y64 = torch.nn.functional.conv2d(x.double(), Wd, padding=1)
    ref = torch.autograd.grad(y64, Wd, dy.double())[0] * k4
    own = torch.zeros_like(bad)
    own[:, c0] = True
    own &= k4 & ~bad
    err = (dW.reshape(ref.shape).double() - ref)[own]
    assert own.any() and (err.norm() / ref[own].norm()).item() <= 2.5e-7
    y = pc.forward(xi, None, relu=False)
    yr = torch.nn.functional.conv2d(x.double(), W.double() * k4, padding=1)
    got = torch.isfinite(y[70, :, :2, :2])
    for h in range(2):
        for w in range(2):  # output (h, w) reads the corner through tap (1 - h, 1 - w)
            assert torch.equal(got[:, h, w], ~(k4 & (W != 0))[:, c0, 1 - h, 1 - w])
    fin = torch.isfinite(y)
    err = (y.double() - yr)[70][fin[70]]
    assert (err.norm() / yr[70][fin[70]].norm()).item() <= 7e-7 and sadmm.device_status() == 0
    if pc.plan.gx_mode:
        e = (y.double() - yr)[70, :, :2, :2][got]
        assert e.numel() == 0 or (e.norm() / yr[70, :, :2, :2][got].norm()).item() <= 7e-7
