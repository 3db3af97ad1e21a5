"""GPU parity of the stride-1 backward on the padded pixel grid (dW, db and dx as
slab GEMMs over shifted copies of x and dZ): shapes at the edges of its tilings
against the fp64 oracle, determinism of every output, and infinities, which
reach exactly the entries whose kept terms hold them.

Tolerances: assert_close's 2e-3 of the largest reference value, as in every
parity test of this suite; the sums are fp32 sums of exact bf16 products."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from workloads import ConvShape

from _helpers import assert_close

pytestmark = pytest.mark.gpu

CASES = [
    # one pixel tile, one channel, seven kernel columns per MMA; resident weights
    ("c1_7x7", ConvShape(n=1, c=1, h=9, w=12, f=16, kh=7, kw=7, ph=3, pw=3), 1.0, wl.COL_SHAPE, 0.6),
    # no pad, more than 16 chunks of channels (two M blocks, the second short), three column tiles
    ("c280_f40", ConvShape(n=2, c=280, h=8, w=7, f=40, kh=3, kw=3), 0.8, wl.COL_SHAPE, 0.3),
    # several filter tiles of dW and long accumulation chains (streamed weights) of dx
    ("c40_f300_groups2", ConvShape(n=3, c=80, h=10, w=10, f=600, kh=3, kw=3, ph=1, pw=1, groups=2), 0.9, wl.COL_SHAPE, 0.5),
    # kernel rows of four taps (no unrolled row), pads of K-1 and of 0, a width below the kernel's
    ("2x4_wide_pad", ConvShape(n=5, c=24, h=6, w=3, f=24, kh=2, kw=4, ph=1, pw=3), 1.0, wl.COL_SHAPE, 0.7),
    ("1x1", ConvShape(n=4, c=72, h=13, w=11, f=136, kh=1, kw=1), 0.5, wl.COL_CHANNEL, 0.5),
    # pixel ranges of several tiles and two pixel tiles per item
    ("many_tiles", ConvShape(n=96, c=32, h=14, w=14, f=96, kh=3, kw=3, ph=1, pw=1), 0.7, wl.COL_CHANNEL, 0.6),
    ("many_tiles_5x5", ConvShape(n=48, c=20, h=19, w=17, f=40, kh=5, kw=5, ph=2, pw=2, groups=2), 0.6, wl.COL_SHAPE, 0.5),
    ("3d_5x3x3", ConvShape(n=3, c=20, t=6, h=7, w=9, f=36, kt=5, kh=3, kw=3, pt=2, ph=1, pw=0), 0.8, wl.COL_NONE, 1.0),
]


def _layer(s, ff, ck, cf, seed):
    from paper_1807_11091_gb300 import sadmm
    dev = torch.device("cuda", 0)
    G = s.cg if ck == wl.COL_CHANNEL else s.k
    kf, kc = wl.retained(ff, s.f), (wl.retained(cf, G) if ck != wl.COL_NONE else 0)
    t = wl.gen_tensors(s, seed=seed)
    rows, cols, _, _ = oracle.project(t["W"], s.taps, kf, ck, kc)
    fi = torch.as_tensor(rows, dtype=torch.int32, device=dev)
    ci = torch.as_tensor(cols, dtype=torch.int32, device=dev) if ck != wl.COL_NONE else None
    pc = sadmm.PrunedConv(s.desc16(), t["W"].to(dev), fi if kf < s.f else None, ck, ci, kf,
                          kc if ck != wl.COL_NONE else s.k)
    g = torch.Generator().manual_seed(seed)
    y = torch.relu(torch.randn(s.y_shape(), generator=g))
    dy = torch.randn(s.y_shape(), generator=g).to(torch.bfloat16)
    return pc, t, rows, cols, y, dy


@pytest.mark.parametrize("case", CASES, ids=lambda c: c[0])
@pytest.mark.parametrize("ydt,relu", [(torch.float32, True), (torch.bfloat16, True), (torch.float32, False)],
                         ids=["y_fp32", "y_bf16", "no_relu"])
def test_grid_backward_matches_oracle(case, ydt, relu):
    from paper_1807_11091_gb300 import sadmm
    name, s, ff, ck, cf = case
    pc, t, rows, cols, y, dy = _layer(s, ff, ck, cf, seed=41)
    y = y.to(ydt).float()
    dev = torch.device("cuda", 0)
    args = (t["x"].to(dev), dy.to(dev))
    dW, db, dx = pc.backward(*args, y=y.to(ydt).to(dev), relu=relu)
    assert sadmm.device_status() == 0
    rdx, rdW, rdb = oracle.pruned_conv_backward(t["x"], t["W"], t["bias"], s.desc16(), s.taps, rows, ck, cols, dy,
                                                relu=relu, y=y)
    rdW = rdW.reshape(s.f, -1)
    assert_close(dW.cpu().numpy(), rdW, what=f"{name} dW")
    assert_close(db.cpu().numpy(), rdb, what=f"{name} db")
    assert_close(dx.cpu().numpy(), rdx, what=f"{name} dx")
    assert np.all(dW.cpu().numpy()[rdW == 0.0] == 0.0)
    again = pc.backward(*args, y=y.to(ydt).to(dev), relu=relu)
    assert all(torch.equal(p, q) for p, q in zip((dW, db, dx), again))


@pytest.mark.parametrize("ck,cf", [(wl.COL_SHAPE, 0.4), (wl.COL_CHANNEL, 0.5)], ids=["shape", "channel"])
def test_infinities_reach_the_kept_terms_alone(ck, cf):
    """An infinity in dY (kept filter, active output) makes the dx entries whose
    kept (channel, tap) read it non-finite and no others; one in x the dW entries
    of its channel, and nothing in dx."""
    from paper_1807_11091_gb300 import sadmm
    s = ConvShape(n=3, c=16, h=9, w=8, f=24, kh=3, kw=3, ph=1, pw=1)
    pc, t, rows, cols, y, dy = _layer(s, 0.5, ck, cf, seed=9)
    dev = torch.device("cuda", 0)
    keep = np.zeros((s.c, s.taps), dtype=bool)
    for c in np.asarray(cols):
        if ck == wl.COL_CHANNEL:
            keep[c] = True
        else:
            keep.reshape(-1)[c] = True
    n0, f0, h0, w0 = 1, int(rows[3]), 4, 2
    y[n0, f0, h0, w0] = 1.0
    dyi = dy.clone()
    dyi[n0, f0, h0, w0] = float("inf")
    W = t["W"].float().numpy().reshape(s.f, s.c, 3, 3)
    want = np.zeros((s.n, s.c, s.h, s.w), dtype=bool)
    for c in range(s.c):
        for kh in range(3):
            for kw in range(3):
                if keep[c, kh * 3 + kw] and W[f0, c, kh, kw] != 0.0:
                    want[n0, c, h0 - 1 + kh, w0 - 1 + kw] = True
    clean = pc.backward(t["x"].to(dev), dy.to(dev), y=y.to(dev))
    dW, db, dx = pc.backward(t["x"].to(dev), dyi.to(dev), y=y.to(dev))
    got = ~torch.isfinite(dx).cpu().numpy()
    assert np.array_equal(got, want)
    assert_close(dx.cpu().numpy()[~want], clean[2].cpu().double().numpy()[~want], tol=1e-6, what="finite dx")
    bad = ~torch.isfinite(dW).cpu().numpy().reshape(s.f, s.c, s.taps)
    assert bad[f0].any() and not bad[np.arange(s.f) != f0].any() and not bad[f0][~keep].any()
    assert not np.isfinite(db.cpu().numpy()[f0]) and np.isfinite(np.delete(db.cpu().numpy(), f0)).all()
    # the corner pixel: taps that would read it from outside the output stay finite
    c0 = int(np.argmax(keep.all(1))) if ck == wl.COL_CHANNEL else int(np.argmax(keep.sum(1)))
    xi = t["x"].clone()
    xi[2, c0, 0, 0] = float("inf")
    dW2, _, dx2 = pc.backward(xi.to(dev), dy.to(dev), y=y.to(dev))
    bad = ~torch.isfinite(dW2).cpu().numpy().reshape(s.f, s.c, 3, 3)
    seen = np.zeros((s.c, 3, 3), dtype=bool)  # x[0, 0] is read by output (1-kh, 1-kw), inside for kh, kw <= 1
    seen[c0, :2, :2] = keep[c0].reshape(3, 3)[:2, :2]
    assert not bad[:, ~seen].any() and bad[np.asarray(rows)][:, seen].all()
    assert torch.equal(dx2, clean[2]) and sadmm.device_status() == 0


@pytest.mark.parametrize("case", [
    ("3x3", ConvShape(n=3, c=16, h=9, w=8, f=24, kh=3, kw=3, ph=1, pw=1)),
    ("no_pad_5x3", ConvShape(n=2, c=20, h=9, w=8, f=40, kh=5, kw=3, groups=2)),
    ("3d", ConvShape(n=2, c=8, t=4, h=5, w=6, f=16, kt=3, kh=3, kw=3, pt=1, ph=1, pw=1)),
], ids=lambda c: c[0])
def test_infinite_weight_reaches_real_outputs_alone(case):
    """dx of a kept weight that is infinite: non-finite where that tap reads an output pixel,
    and the sum of the other terms where it would read one past the output's edge."""
    from paper_1807_11091_gb300 import sadmm
    name, s = case
    dev = torch.device("cuda", 0)
    g = torch.Generator().manual_seed(3)
    W = torch.randn(s.w_shape(), generator=g).to(torch.bfloat16)
    x = torch.randn(s.x_shape(), generator=g).to(torch.bfloat16)
    dy = (torch.rand(s.y_shape(), generator=g) + 0.5).to(torch.bfloat16)
    f0, c0, tap = 3, 1, 0  # conv group 0, the first tap: reads output (t + pt, h + ph, w + pw)
    cols = np.sort(np.random.default_rng(1).permutation(s.k)[:s.k // 2])
    cols = np.unique(np.append(cols, c0 * s.taps + tap))
    mask = np.zeros(s.k, dtype=bool)
    mask[cols] = True
    Wm = (W.double().reshape(s.f, s.k) * torch.from_numpy(mask)).reshape(W.shape)
    Wf = Wm.clone()
    Wf.reshape(s.f, s.k)[f0, c0 * s.taps + tap] = 0.0
    conv = torch.nn.functional.conv3d if s.is3d else torch.nn.functional.conv2d
    pad = (s.pt, s.ph, s.pw) if s.is3d else (s.ph, s.pw)
    xd = x.double().requires_grad_(True)
    want, = torch.autograd.grad(conv(xd, Wf, padding=pad, groups=s.groups), xd, dy.double())
    W.reshape(s.f, s.k)[f0, c0 * s.taps + tap] = float("inf")
    t, h, w = np.meshgrid(np.arange(s.t), np.arange(s.h), np.arange(s.w), indexing="ij")
    real = (t + s.pt < s.ot) & (h + s.ph < s.oh) & (w + s.pw < s.ow)
    bad = np.zeros((s.n, s.c, s.t, s.h, s.w), dtype=bool)
    bad[:, c0] = real
    bad = bad.reshape(x.shape)
    ci = torch.as_tensor(cols, dtype=torch.int32, device=dev)
    pc = sadmm.PrunedConv(s.desc16(), W.to(dev), None, wl.COL_SHAPE, ci, s.f, len(cols))
    dW, db, dx = pc.backward(x.to(dev), dy.to(dev), relu=False)
    got = dx.cpu().double().numpy()
    assert sadmm.device_status() == 0
    assert np.array_equal(~np.isfinite(got), bad)
    ref = want.numpy()
    assert np.abs(got[~bad] - ref[~bad]).max() <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("case", [
    # stages longer than a segment: cut at kernel rows, and inside one
    ("7x7", ConvShape(n=4, c=32, h=28, w=28, f=64, kh=7, kw=7, ph=3, pw=3)),
    ("11x11", ConvShape(n=4, c=32, h=20, w=20, f=64, kh=11, kw=11, ph=5, pw=5)),
    ("1x31", ConvShape(n=8, c=16, h=4, w=96, f=32, kh=1, kw=31, ph=0, pw=15)),
    # unrolled rows, one and two 16-filter groups a stage
    ("5x5", ConvShape(n=4, c=48, h=27, w=27, f=72, kh=5, kw=5, ph=2, pw=2)),
    ("3x3", ConvShape(n=4, c=64, h=28, w=28, f=64, kh=3, kw=3, ph=1, pw=1)),
    ("3d", ConvShape(n=2, c=16, t=6, h=14, w=14, f=64, kt=3, kh=3, kw=3, pt=1, ph=1, pw=1)),
    # long sums over the filters
    ("512_filters", ConvShape(n=8, c=32, h=9, w=9, f=512, kh=3, kw=3, ph=1, pw=1)),
], ids=lambda c: c[0])
def test_input_gradient_error_against_64_bits(case):
    """dx in the 2-norm against 64 bits: the tensor core truncates about 1e-8 of a sum per
    step of 16, and its sums are cut after 12 steps (27 past 256 filters); the fp32 additions
    of the at most 130 segments add about 1e-7.  Uncut, the 7x7 and 11x11 layers stand at 4
    to 12e-7."""
    from paper_1807_11091_gb300 import sadmm
    name, s = case
    dev = torch.device("cuda", 0)
    g = torch.Generator().manual_seed(8)
    W = (torch.randn(s.w_shape(), generator=g) * 0.1).to(torch.bfloat16).to(dev)
    x = torch.relu(torch.randn(s.x_shape(), generator=g)).to(torch.bfloat16).to(dev)
    dy = torch.randn(s.y_shape(), generator=g).to(torch.bfloat16).to(dev)
    pc = sadmm.PrunedConv(s.desc16(), W, None, wl.COL_NONE, None, s.f, s.k)
    dx = pc.backward(x, dy, relu=False)[2]
    assert sadmm.device_status() == 0
    conv = torch.nn.functional.conv3d if s.is3d else torch.nn.functional.conv2d
    xd = x.double().requires_grad_(True)
    ref, = torch.autograd.grad(conv(xd, W.double(), padding=(s.pt, s.ph, s.pw) if s.is3d else (s.ph, s.pw)), xd, dy.double())
    assert ((dx.double() - ref).norm() / ref.norm()).item() <= (3.5e-7 if s.f > 256 else 2.5e-7)
