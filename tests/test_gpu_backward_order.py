"""The pixel-grid backward's launches overlap (the input gradient starts beside the
weight gradient's last items and waits for it at its end): calls issued back to
back, and replayed from a CUDA graph, on one reused workspace give bit for bit what
calls with the device idle in between give."""
import pytest
import torch

import workloads as wl
from workloads import ConvShape

pytestmark = pytest.mark.gpu

SHAPES = [
    ConvShape(n=1, c=8, h=6, w=6, f=8, kh=3, kw=3, ph=1, pw=1),  # one item each, small shared memory
    ConvShape(n=24, c=48, h=27, w=27, f=64, kh=5, kw=5, ph=2, pw=2),  # several rounds of weight-gradient items
    ConvShape(n=16, c=64, h=28, w=28, f=64, kh=1, kw=1),  # input gradient short beside the weight gradient
]


@pytest.mark.parametrize("s", SHAPES, ids=["tiny", "5x5", "1x1"])
@pytest.mark.parametrize("graph", [False, True], ids=["stream", "graph"])
def test_back_to_back_calls(s, graph):
    from paper_1807_11091_gb300 import sadmm
    dev = torch.device("cuda", 0)
    g = torch.Generator().manual_seed(5)
    W = torch.randn(s.f, s.k, generator=g).to(torch.bfloat16).to(dev)
    kf, kc = s.f // 2, max(1, s.k // 2)
    fi, ci, _ = sadmm.project_groups(s.desc16(), W, kf, wl.COL_SHAPE, kc)
    pc = sadmm.PrunedConv(s.desc16(), W, fi, wl.COL_SHAPE, ci, kf, kc)
    xs = [torch.randn(s.n, s.c, s.h, s.w, generator=g).to(torch.bfloat16).to(dev) for _ in range(2)]
    dys = [torch.randn(s.y_shape(), generator=g).to(torch.bfloat16).to(dev) for _ in range(2)]
    want = []
    for x, dy in zip(xs, dys):
        want.append([t.clone() for t in pc.backward(x, dy, relu=False)])
        torch.cuda.synchronize()
    if graph:
        run = torch.cuda.CUDAGraph()
        x, dy = xs[0].clone(), dys[0].clone()
        with torch.cuda.graph(run):
            a = pc.backward(x, dy, relu=False)
            b = pc.backward(x, dy, relu=False)
        for i in (0, 1, 0, 1):
            x.copy_(xs[i])
            dy.copy_(dys[i])
            run.replay()
            assert all(torch.equal(p, q) for out in (a, b) for p, q in zip(out, want[i]))
    else:
        got = [[t.clone() for t in pc.backward(xs[i & 1], dys[i & 1], relu=False)] for i in range(12)]
        for i, out in enumerate(got):
            assert all(torch.equal(p, q) for p, q in zip(out, want[i & 1]))
    assert sadmm.device_status() == 0


def test_rejected_lists_without_a_bias_gradient():
    """A plan whose index lists pack rejected keeps no filter: with no bias gradient every
    block of the slice reduction returns early.  The launch still ends after the input
    gradient's, so what follows on the stream reads every dx written: zeros, back to back."""
    from paper_1807_11091_gb300 import sadmm
    dev = torch.device("cuda", 0)
    s = ConvShape(n=64, c=48, h=27, w=27, f=64, kh=5, kw=5, ph=2, pw=2)
    g = torch.Generator().manual_seed(6)
    W = torch.randn(s.f, s.k, generator=g).to(torch.bfloat16).to(dev)
    fi = torch.arange(s.f // 2, dtype=torch.int32, device=dev)
    ci = torch.arange(s.k // 2, dtype=torch.int32, device=dev)
    pc = sadmm.PrunedConv(s.desc16(), W, fi, wl.COL_SHAPE, ci, s.f // 2, s.k // 2)
    fi[3] = s.f
    pc.repack(W, fi, ci)
    assert sadmm.device_status() == sadmm.SADMM_EINVAL
    x = torch.randn(s.n, s.c, s.h, s.w, generator=g).to(torch.bfloat16).to(dev)
    dy = torch.randn(s.y_shape(), generator=g).to(torch.bfloat16).to(dev)
    need = sadmm.sadmm_conv_bwd_workspace_size(pc.plan)
    ws = torch.empty(need + 1024, dtype=torch.uint8, device=dev)
    at = (ws.data_ptr() + 1023) // 1024 * 1024
    dW = torch.empty(s.f, s.k, device=dev)
    dx = torch.empty(x.shape, device=dev)
    seen = []
    for _ in range(6):
        dW.fill_(1.0)
        dx.fill_(1.0)
        st = sadmm.sadmm_conv_bwd(pc.plan, x.data_ptr(), dy.data_ptr(), None, sadmm.SADMM_FP32, 0, dW.data_ptr(), None,
                                  dx.data_ptr(), at, need, int(torch.cuda.current_stream().cuda_stream))
        assert st == 0
        seen += [dW.clone(), dx.clone()]
    assert all(not t.any() for t in seen) and sadmm.device_status() == 0
