"""The binding launches on the current device's current stream, as
torch.cuda.current_stream() names it, or on the stream it is given."""
import pytest
import torch

import workloads as wl
from workloads import ConvShape

pytestmark = pytest.mark.gpu


def test_current_stream_and_given_stream():
    from paper_1807_11091_gb300 import sadmm
    dev = torch.device("cuda", 0)
    s = ConvShape(n=1, c=8, h=9, w=9, f=16, kh=3, kw=3, ph=1, pw=1)
    t = wl.gen_tensors(s, seed=1)
    pc = sadmm.PrunedConv(s.desc16(), t["W"].to(dev), None, wl.COL_NONE, None, s.f, s.k)
    x, bias = t["x"].to(dev), t["bias"].to(dev)
    ref = pc.forward(x, bias)
    torch.cuda.synchronize()
    assert sadmm._stream() == int(torch.cuda.current_stream().cuda_stream)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert sadmm._stream() == int(side.cuda_stream)
        y = pc.forward(x, bias)
    side.synchronize()
    assert torch.equal(y, ref)
    y2 = torch.empty_like(ref)
    side.wait_stream(torch.cuda.current_stream())
    pc.forward(x, bias, out=y2, stream=side)
    side.synchronize()
    assert torch.equal(y2, ref)
