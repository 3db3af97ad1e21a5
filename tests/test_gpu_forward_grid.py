"""GPU parity of the forward on the padded pixel grid (plan.gx_mode = 1): layers
the rule sends there, at the edges of its tilings, against the fp64 oracle;
which layers it takes; capped plans; infinities, which reach exactly the outputs
whose kept terms hold them; and index lists a pack rejects.

Tolerances: assert_close's 2e-3 of the largest reference value (fp32 sums of
exact bf16 products), and half a unit in the last place of bf16 more for bf16
outputs."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from workloads import ConvShape

from _helpers import assert_close

pytestmark = pytest.mark.gpu

CASES = [
    # resident weights, a ragged last tile, pruned filters' planes
    ("c62_f48", ConvShape(n=3, c=62, h=99, w=101, f=48, kh=3, kw=3, ph=1, pw=1), 0.7, wl.COL_SHAPE, 0.9),
    # three groups of unequal kept counts, 5x5
    ("groups3_5x5", ConvShape(n=3, c=48, h=57, w=53, f=72, kh=5, kw=5, ph=2, pw=2, groups=3), 0.5, wl.COL_SHAPE, 0.6),
    # weights in a ring, several column tiles, no pad
    ("c96_f280", ConvShape(n=1, c=96, h=145, w=145, f=280, kh=3, kw=3), 1.0, wl.COL_SHAPE, 1.0),
    # channel-wise pruning, kernel rows of seven taps (no unrolled row), asymmetric pads
    ("channel_3x7", ConvShape(n=2, c=160, h=101, w=100, f=64, kh=3, kw=7, ph=2, pw=1), 0.9, wl.COL_CHANNEL, 0.5),
    # frames
    ("video", ConvShape(n=2, c=32, t=5, h=45, w=44, f=64, kt=3, kh=3, kw=3, pt=1, ph=1, pw=1), 1.0, wl.COL_SHAPE, 0.95),
]


def _packed(s, ff, ck, cf, seed=29, max_ctas=0):
    from paper_1807_11091_gb300 import sadmm
    dev = torch.device("cuda", 0)
    G = s.cg if ck == wl.COL_CHANNEL else s.k
    kf, kc = wl.retained(ff, s.f), wl.retained(cf, G)
    t = wl.gen_tensors(s, seed=seed)
    rows, cols, _, _ = oracle.project(t["W"], s.taps, kf, ck, kc)
    fi = torch.as_tensor(rows, dtype=torch.int32, device=dev)
    ci = torch.as_tensor(cols, dtype=torch.int32, device=dev)
    pc = sadmm.PrunedConv(s.desc16(), t["W"].to(dev), fi if kf < s.f else None, ck, ci, kf, kc, max_ctas=max_ctas)
    return pc, t, rows, cols


@pytest.mark.parametrize("case", CASES, ids=lambda c: c[0])
def test_grid_forward_matches_oracle(case):
    from paper_1807_11091_gb300 import sadmm
    name, s, ff, ck, cf = case
    pc, t, rows, cols = _packed(s, ff, ck, cf)
    assert pc.plan.gx_mode == 1
    dev = torch.device("cuda", 0)
    x, bias = t["x"].to(dev), t["bias"].to(dev)
    ref = oracle.pruned_conv(t["x"], t["W"], t["bias"], s.desc16(), s.taps, rows, ck, cols, relu=True)
    y = pc.forward(x, bias)
    yh = pc.forward(x, bias, out_dtype=torch.bfloat16)
    assert sadmm.device_status() == 0
    assert_close(y.cpu().numpy(), ref, what=name)
    assert torch.equal(yh, y.to(torch.bfloat16))  # one rounding of the same sums
    assert torch.equal(y, pc.forward(x, bias))
    capped, _, _, _ = _packed(s, ff, ck, cf, max_ctas=37)
    assert torch.equal(y, capped.forward(x, bias))  # the sums do not follow the tiling
    lin = pc.forward(x, None, relu=False)
    ref = oracle.pruned_conv(t["x"], t["W"], torch.zeros_like(t["bias"]), s.desc16(), s.taps, rows, ck, cols, relu=False)
    assert_close(lin.cpu().numpy(), ref, what=f"{name} linear")


def test_which_layers_take_the_grid():
    """Shape-wise layers by density (AlexNet conv2 at half, not conv3 at a
    quarter), and none with a stride, a single tap or few output tiles."""
    from paper_1807_11091_gb300 import sadmm

    def mode(s, ff, ck, cf):
        G = s.cg if ck == wl.COL_CHANNEL else s.k
        st, p = sadmm.sadmm_plan_init(sadmm.make_desc(s.desc16()), wl.retained(ff, s.f), ck, wl.retained(cf, G))
        assert st == 0
        return p.gx_mode
    a = wl.alexnet()
    assert mode(a[1].shape, 0.5, wl.COL_SHAPE, 0.5) == 1 and mode(a[2].shape, 0.25, wl.COL_SHAPE, 0.25) == 0
    assert mode(a[2].shape, 1.0, wl.COL_SHAPE, 1.0) == 1 and mode(a[2].shape.with_batch(8), 1.0, wl.COL_SHAPE, 1.0) == 0
    s = ConvShape(n=8, c=96, h=64, w=64, f=96, kh=3, kw=3, ph=1, pw=1)
    assert mode(s, 1.0, wl.COL_SHAPE, 0.9) == 1
    import dataclasses
    assert mode(dataclasses.replace(s, sh=2, sw=2, n=32), 1.0, wl.COL_SHAPE, 0.9) == 0
    assert mode(dataclasses.replace(s, kh=1, kw=1, ph=0, pw=0), 1.0, wl.COL_SHAPE, 0.9) == 0
    assert mode(dataclasses.replace(s, ph=3), 1.0, wl.COL_SHAPE, 0.9) == 0


def test_infinities_reach_the_kept_terms_alone():
    from paper_1807_11091_gb300 import sadmm
    s = ConvShape(n=3, c=64, h=100, w=100, f=32, kh=3, kw=3, ph=1, pw=1)
    pc, t, rows, cols = _packed(s, 0.75, wl.COL_SHAPE, 0.8)
    assert pc.plan.gx_mode == 1
    dev = torch.device("cuda", 0)
    keep = np.zeros((s.c, 3, 3), dtype=bool)
    keep.reshape(-1)[np.asarray(cols)] = True
    c0 = int(np.argmin(np.where(keep.reshape(s.c, -1).any(1), keep.reshape(s.c, -1).sum(1), 99)))
    clean = pc.forward(t["x"].to(dev), t["bias"].to(dev), relu=False)
    for (n, h, w) in ((1, 0, 99), (0, 50, 31), (1, 99, 0)):
        xi = t["x"].clone()
        xi[n, c0, h, w] = float("inf")
        y = pc.forward(xi.to(dev), t["bias"].to(dev), relu=False)
        want = np.zeros(s.y_shape(), dtype=bool)
        for kh in range(3):
            for kw in range(3):
                oh, ow = h + 1 - kh, w + 1 - kw
                if keep[c0, kh, kw] and 0 <= oh < s.h and 0 <= ow < s.w:
                    want[n, np.asarray(rows), oh, ow] = t["W"][:, c0, kh, kw].float().numpy()[np.asarray(rows)] != 0
        bad = ~torch.isfinite(y).cpu().numpy()
        assert np.array_equal(bad, want)
        # outputs whose pruned taps see the infinity are summed again in another order: fp32 rounding apart
        assert_close(y.cpu().numpy()[~want], clean.cpu().double().numpy()[~want], tol=1e-5, what="finite outputs")
    assert sadmm.device_status() == 0


def test_rejected_lists_give_zeros_and_a_repack_restores():
    from paper_1807_11091_gb300 import sadmm
    s = ConvShape(n=3, c=48, h=100, w=100, f=40, kh=3, kw=3, ph=1, pw=1)
    pc, t, rows, cols = _packed(s, 0.8, wl.COL_SHAPE, 0.9)
    assert pc.plan.gx_mode == 1
    dev = torch.device("cuda", 0)
    x, bias, W = t["x"].to(dev), t["bias"].to(dev), t["W"].to(dev)
    good = pc.forward(x, bias)
    fi = torch.as_tensor(rows, dtype=torch.int32, device=dev)
    ci = torch.as_tensor(cols, dtype=torch.int32, device=dev)
    pc.repack(W, fi, ci.flip(0))
    y = pc.forward(x, bias)
    assert sadmm.device_status() == sadmm.SADMM_EINVAL
    assert torch.equal(y, torch.zeros_like(y))
    pc.repack(W, fi, ci)
    assert torch.equal(pc.forward(x, bias), good) and sadmm.device_status() == 0
