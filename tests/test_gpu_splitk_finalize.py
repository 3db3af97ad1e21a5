"""GPU parity of the split-K' reduction: 16-byte and element-wise pixel runs
(planes of a multiple of four pixels or not, outputs off the 16-byte grid), a
last tile that ends inside a run, several conv groups, and the pruned filters'
zero planes, which the conv kernel's splits write between them.  Tolerance:
assert_close's (fp32 sums of exact bf16 products) and, for bf16 outputs, half a
unit in the last place more."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl
from workloads import ConvShape

from _helpers import assert_close

pytestmark = pytest.mark.gpu

CASES = [
    ("plane64_pruned", ConvShape(n=3, c=40, h=8, w=8, f=70, kh=3, kw=3, ph=1, pw=1), 0.4, 0.8),
    ("plane20_groups3", ConvShape(n=7, c=96, h=5, w=4, f=48, kh=3, kw=3, ph=1, pw=1, groups=3), 0.6, 1.0),
    ("plane49", ConvShape(n=4, c=64, h=7, w=7, f=300, kh=3, kw=3, ph=1, pw=1), 0.3, 0.5),
    ("plane36_one_kept", ConvShape(n=1, c=640, h=6, w=6, f=200, kh=1, kw=1), 0.005, 1.0),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: c[0])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["fp32", "bf16"])
@pytest.mark.parametrize("shift", [0, 1], ids=["aligned", "one_element_off"])
def test_split_reduction(case, dtype, shift):
    from paper_1807_11091_gb300 import sadmm
    name, s, ff, cf = case
    dev = torch.device("cuda", 0)
    kf, kc = wl.retained(ff, s.f), wl.retained(cf, s.k)
    t = wl.gen_tensors(s, seed=3)
    rows, cols, _, _ = oracle.project(t["W"], s.taps, kf, wl.COL_SHAPE, kc)
    fi = torch.as_tensor(rows, dtype=torch.int32, device=dev)
    ci = torch.as_tensor(cols, dtype=torch.int32, device=dev)
    pc = sadmm.PrunedConv(s.desc16(), t["W"].to(dev), fi, wl.COL_SHAPE, ci, kf, kc)
    assert pc.plan.splits > 1
    ref = oracle.pruned_conv(t["x"], t["W"], t["bias"], s.desc16(), s.taps, rows, wl.COL_SHAPE, cols, relu=True)
    buf = torch.full((int(np.prod(s.y_shape())) + 8,), float("nan"), dtype=dtype, device=dev)
    y = buf[shift:shift + int(np.prod(s.y_shape()))].view(s.y_shape())
    pc.forward(t["x"].to(dev), t["bias"].to(dev), out=y)
    assert sadmm.device_status() == 0
    got = y.float().cpu().numpy()
    assert_close(got, ref, tol=2e-3 if dtype == torch.float32 else 2e-3 + 2.0 ** -8, what=f"{name} {dtype}")
    pruned = np.setdiff1d(np.arange(s.f), rows)
    assert np.all(got[:, pruned] == 0.0)
    assert torch.isnan(buf[:shift].float()).all() and torch.isnan(buf[shift + y.numel():].float()).all()
