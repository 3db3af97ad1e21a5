"""The work a user of this library has it do, as timed cases.

A program that serves or retrains a structurally pruned network (StructADMM,
arXiv 1807.11091) calls four things over and over: the pruned CONV forward,
the masked-retraining backward, the ADMM Z/U update, and, when masks change,
the projection and pack of every layer followed by its forward.  Each case is
one such pass through the public entry points (``sadmm.PrunedConv``,
``sadmm.AdmmBatch``, ``sadmm.ProjectBatch``, ``sadmm.pack_batch``).  Layer
shapes and densities are those of ``workloads.py``; ``draw`` varies them.

A case's ``op`` is one of
  fwd   one packed layer, forward: x (bf16) -> y (fp32 or bf16)
  bwd   one packed layer, backward: dY (bf16) and the forward's y -> dW, db, dx
  admm  one ADMM update of every layer of a network: W, U -> Z, U, kept lists
  net   projection, pack and forward of every layer of a network (new masks)
"""
import math

import torch

import workloads as wl
from paper_1807_11091_gb300 import sadmm

SHAPE_KEYS = ("n", "c", "t", "h", "w", "f", "groups", "kt", "kh", "kw", "st", "sh", "sw", "pt", "ph", "pw")


# ------------------------------------------------------------------ cases --

def _layer_case(name, op, layer, n=None, relu=True, out="fp32", dx=True):
    s = layer.shape if n is None else layer.shape.with_batch(n)
    c = {"name": name, "op": op}
    c.update(zip(SHAPE_KEYS, s.desc16()))
    c.update(filt_frac=layer.filt_frac, colkind=layer.colkind, col_frac=layer.col_frac, relu=relu, out=out, dx=dx)
    return c


def listed():
    a = wl.alexnet()
    r = {L.name: L for L in wl.resnet50()}
    return [
        # one image through one layer: the paper's own timing setting, where launches and start-up count
        _layer_case("fwd_alexnet_conv3_b1", "fwd", a[2], n=1),
        # a small layer at a small batch, half of the columns kept
        _layer_case("fwd_small2d_b8", "fwd", wl.single2d()[0]),
        # a network's first layer: 3 channels, 11x11 stride 4, kept whole; the largest output of its network
        _layer_case("fwd_alexnet_conv1_b128", "fwd", a[0]),
        # grouped 5x5, half of the filters and half of the columns, odd 27x27 planes
        _layer_case("fwd_alexnet_conv2_b128", "fwd", a[1]),
        # 1x1 with half of the channels, few columns and a large output; written in bf16 for the next layer
        _layer_case("fwd_resnet_1x1_b64", "fwd", r["r56_64x256_1x1"], out="bf16"),
        # video: 3-D taps, 30 % of the columns
        _layer_case("fwd_video3d_b8", "fwd", wl.c3d()[0]),
        # the widest layer and largest contraction, half of the columns
        _layer_case("fwd_wide_b128", "fwd", wl.sweep((0.5,), (1.0,))[0]),
        # retraining steps: 13x13 planes at a quarter of the weights per dimension,
        _layer_case("bwd_alexnet_conv3_b128", "bwd", a[2]),
        # grouped 5x5 at half (the costliest backward of its network),
        _layer_case("bwd_alexnet_conv2_b128", "bwd", a[1]),
        # and a bottleneck 3x3 with half of the channels
        _layer_case("bwd_resnet_3x3_b64", "bwd", r["r28_128x128_3x3"]),
        # one ADMM iteration's update of all five layers, training precision
        {"name": "admm_alexnet", "op": "admm", "net": "alexnet", "dtype": "fp32", "keep": 1.0},
        # new masks for a whole network: 16 projections, 16 packs, 16 forwards
        {"name": "net_resnet50_b64", "op": "net", "net": "resnet50", "n": 64, "keep": 1.0},
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.random()
    if kind < 0.08:
        return {"op": "admm", "net": rng.choice(["alexnet", "resnet50"]), "dtype": rng.choice(["fp32", "bf16"]),
                "keep": round(rng.uniform(0.3, 1.0), 3)}
    if kind < 0.16:
        return {"op": "net", "net": rng.choice(["alexnet", "resnet50"]), "n": _logint(rng, 1, 32),
                "keep": round(rng.uniform(0.5, 1.0), 3)}
    op = "fwd" if kind < 0.62 else "bwd"
    while True:
        k = rng.choice([1, 3, 3, 3, 5])
        video = k == 3 and rng.random() < 0.15
        groups = rng.choice([1, 1, 1, 2])
        s = rng.choice([1, 1, 1, 1, 2])
        h = _logint(rng, 7, 112)
        w = h if rng.random() < 0.7 else _logint(rng, 7, 112)
        pad = k // 2 if rng.random() < 0.85 else 0
        c = {"op": op, "n": _logint(rng, 1, 128), "c": groups * _logint(rng, 3, 512), "t": _logint(rng, 2, 16) if video else 1,
             "h": h, "w": w, "f": groups * _logint(rng, 16, 512), "groups": groups, "kt": 3 if video else 1, "kh": k, "kw": k,
             "st": 1, "sh": s, "sw": s, "pt": 1 if video else 0, "ph": pad, "pw": pad}
        colkind = rng.choice([wl.COL_SHAPE, wl.COL_SHAPE, wl.COL_CHANNEL, wl.COL_NONE])
        c.update(filt_frac=round(rng.choice([1.0, rng.uniform(0.15, 1.0)]), 3), colkind=colkind,
                 col_frac=1.0 if colkind == wl.COL_NONE else round(rng.uniform(0.1, 1.0), 3),
                 relu=rng.random() < 0.8, out=rng.choice(["fp32", "fp32", "bf16"]), dx=rng.random() < 0.85)
        L = _layer(c)
        sh = L.shape
        if sh.oh < 1 or sh.ow < 1 or sh.k > 8192 or L.k_filters < 1 or L.k_cols < 1:
            continue
        # no costlier than the listed cases: input and output elements, pixels x kept columns, multiply-adds
        lim = 1.0 if op == "fwd" else 0.5
        if (sh.n * sh.c * sh.t * sh.h * sh.w <= lim * 2.6e7 and sh.m * sh.f <= lim * 5.1e7
                and sh.m * sh.groups * L.n_cols <= lim * 1.1e8 and sh.m * L.k_filters * L.n_cols <= lim * 5.9e10):
            return c


# ----------------------------------------------------------------- inputs --

def _layer(c):
    s = wl.ConvShape(**{k: c[k] for k in SHAPE_KEYS})
    return wl.Layer("case", s, c["filt_frac"], c["colkind"], c["col_frac"], seed=0)


def _net(c):
    """The layers of a network case: its own densities times `keep`, its own batch."""
    import dataclasses
    out = []
    for L in wl.get(c["net"]):
        s = L.shape.with_batch(c["n"]) if "n" in c else L.shape
        out.append(dataclasses.replace(L, shape=s, filt_frac=max(L.filt_frac * c["keep"], 1.0 / s.f),
                                       col_frac=max(L.col_frac * c["keep"], 1.0 / L.col_groups)))
    return out


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _weights(s, g):
    """He-initialised weights in fp32 and a bias of standard deviation 0.1."""
    W = torch.randn(s.w_shape(), generator=g, device="cuda") * math.sqrt(2.0 / (s.cg * s.taps))
    return W, torch.randn(s.f, generator=g, device="cuda") * 0.1


def _input(s, g):
    return torch.relu(torch.randn(s.x_shape(), generator=g, device="cuda")).to(torch.bfloat16)


def _layer_inputs(c, seed):
    """W (bf16), bias, x and, for a backward, dY and the forward's output y."""
    L = _layer(c)
    s, g = L.shape, _gen(seed)
    W, bias = _weights(s, g)
    W, x = W.to(torch.bfloat16), _input(s, g)
    if c["op"] == "fwd":
        return L, W, bias, x, None, None
    dy = (torch.randn(s.y_shape(), generator=g, device="cuda") * 0.01).to(torch.bfloat16)
    y = torch.relu(torch.randn(s.y_shape(), generator=g, device="cuda"))  # about half of the outputs are active
    return L, W, bias, x, dy, (y.to(torch.bfloat16) if c["out"] == "bf16" else y)


def _admm_inputs(c, seed):
    dt = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    g = _gen(seed)
    Ws, Us = [], []
    for L in _net(c):
        sd = math.sqrt(2.0 / (L.shape.cg * L.shape.taps))
        Ws.append((torch.randn(L.shape.w_shape(), generator=g, device="cuda") * sd).to(dt))
        Us.append((torch.randn(L.shape.w_shape(), generator=g, device="cuda") * (sd * math.sqrt(0.1))).to(dt))
    return Ws, Us


def _net_inputs(c, seed):
    g, out = _gen(seed), []
    for L in _net(c):
        W, bias = _weights(L.shape, g)
        out.append((L, W.to(torch.bfloat16), bias, _input(L.shape, g)))
    return out


def _pack(L, W):
    d = L.shape.desc16()
    fi, ci, _ = sadmm.project_groups(d, W, L.k_filters, L.colkind, 0 if L.colkind == wl.COL_NONE else L.k_cols)
    return sadmm.PrunedConv(d, W, fi, L.colkind, ci, L.k_filters, L.k_cols)


def prepare(case, seed):
    """Inputs on the GPU and what a program keeps: packed layers, batch handles."""
    if case["op"] in ("fwd", "bwd"):
        L, W, bias, x, dy, y = _layer_inputs(case, seed)
        return {"case": case, "pc": _pack(L, W), "bias": bias, "x": x, "dy": dy, "y": y}
    if case["op"] == "admm":
        Ws, Us = _admm_inputs(case, seed)
        specs = [(L.shape.desc16(), L.k_filters, L.colkind, L.k_cols) for L in _net(case)]
        return {"case": case, "step": sadmm.AdmmBatch(specs, Ws[0].device), "W": Ws, "U": Us,
                "Z": [torch.empty_like(W) for W in Ws]}
    items = _net_inputs(case, seed)
    proj = sadmm.ProjectBatch([(L.shape.desc16(), W, L.k_filters, L.colkind, L.k_cols, None) for L, W, _, _ in items])
    return {"case": case, "proj": proj, "items": items, "convs": [_pack(L, W) for L, W, _, _ in items]}


def run(state):
    c = state["case"]
    if c["op"] == "fwd":
        out = torch.bfloat16 if c["out"] == "bf16" else torch.float32
        return state["pc"].forward(state["x"], state["bias"], relu=c["relu"], out_dtype=out)
    if c["op"] == "bwd":
        dW, db, dx = state["pc"].backward(state["x"], state["dy"], y=state["y"] if c["relu"] else None, relu=c["relu"],
                                          want_dx=c["dx"])
        return {"dW": dW, "db": db, "dx": dx} if c["dx"] else {"dW": dW, "db": db}
    if c["op"] == "admm":
        kept = state["step"](state["W"], state["U"], state["Z"])
        return {"Z": list(state["Z"]), "U": list(state["U"]), "filt": [k[0] for k in kept], "cols": [k[1] for k in kept]}
    kept = state["proj"]()
    sadmm.pack_batch([(pc, W, fi, ci) for pc, (_, W, _, _), (fi, ci, _) in zip(state["convs"], state["items"], kept)])
    ys = [pc.forward(x, bias) for pc, (_, _, bias, x) in zip(state["convs"], state["items"])]
    return {"filt": [k[0] for k in kept], "cols": [k[1] for k in kept], "y": ys}


# ------------------------------------------------------- what a pass needs --

def _fwd_work(L, ysize):
    s = L.shape
    chans = s.groups * L.k_cols if L.colkind == wl.COL_CHANNEL else s.c
    return (2 * s.n * chans * s.t * s.h * s.w + 2 * L.k_filters * L.n_cols + ysize * s.m * s.f + 4 * s.f,
            L.retained_flops())


def work(case):
    if case["op"] == "fwd":
        b, f = _fwd_work(_layer(case), 2 if case["out"] == "bf16" else 4)
        return {"bytes": b, "flops": f}
    if case["op"] == "bwd":
        L = _layer(case)
        s = L.shape
        kept_y = s.m * L.k_filters  # only the kept filters' planes of dY and y matter
        chans = s.groups * L.k_cols if L.colkind == wl.COL_CHANNEL else s.c
        xsize = s.n * s.t * s.h * s.w
        b = 2 * kept_y + (kept_y * (2 if case["out"] == "bf16" else 4) if case["relu"] else 0)
        b += 2 * xsize * chans + 4 * s.f * s.k + 4 * s.f
        f = L.retained_flops()
        if case["dx"]:
            b += 4 * xsize * s.c + 2 * L.k_filters * L.n_cols
            f *= 2
        return {"bytes": b, "flops": f}
    if case["op"] == "admm":
        e = 4 if case["dtype"] == "fp32" else 2
        n = sum(L.shape.f * L.shape.k for L in _net(case))
        return {"bytes": 4 * e * n, "flops": 5 * n}
    b = f = 0
    for L in _net(case):
        lb, lf = _fwd_work(L, 4)
        b += lb + 2 * L.shape.f * L.shape.k
        f += lf
    return {"bytes": b, "flops": f}


def tolerance(case):
    """fp32 results are fp32 sums of exact bf16 products.  Against the 64-bit value the forward shows 7e-8 to 7e-7 at
    4 to 72 tensor-core steps of 16 columns, about 1e-8 per step (2e-6 at the 200 steps the widest drawn layers
    have), and the backward up to 3e-7.  A bf16 result adds its own rounding (1.7e-3).  The ADMM update rounds
    W + U once and then copies, and the kept lists are whole numbers."""
    if case["op"] == "admm":
        return "exact"
    if case["op"] == "fwd" and case["out"] == "bf16":
        return {"rel": 7e-3, "max": 2e-2}
    return {"rel": 1e-5, "max": 2e-4}


# ------------------------------------------------------------ 64-bit values --

def _top(keys, k):
    """Indices of the k largest keys (equal keys: the lower index), ascending."""
    return torch.sort(torch.sort(keys, descending=True, stable=True)[1][:k])[0]


def _kept(L, V):
    """Kept filters and kept column groups of V [F][K]: filters first, then columns over the kept filters."""
    s = L.shape
    sq = V.double().reshape(s.f, s.k) ** 2
    fi = _top(sq.sum(1), L.k_filters)
    if L.colkind == wl.COL_NONE:
        return fi, None, torch.arange(s.k, device=V.device)
    ck = sq[fi].sum(0)
    if L.colkind == wl.COL_SHAPE:
        ci = _top(ck, L.k_cols)
        return fi, ci, ci
    ci = _top(ck.reshape(s.cg, s.taps).sum(1), L.k_cols)
    return fi, ci, (ci[:, None] * s.taps + torch.arange(s.taps, device=V.device)).reshape(-1)


def _mask(L, fi, cols):
    m = torch.zeros(L.shape.f, L.shape.k, dtype=torch.float64, device=fi.device)
    m[fi[:, None], cols[None, :]] = 1.0
    return m


def _conv64(s, x, W):
    if s.is3d:
        return torch.nn.functional.conv3d(x, W, stride=(s.st, s.sh, s.sw), padding=(s.pt, s.ph, s.pw), groups=s.groups)
    return torch.nn.functional.conv2d(x, W, stride=(s.sh, s.sw), padding=(s.ph, s.pw), groups=s.groups)


def _fwd64(L, W, bias, x, relu):
    s = L.shape
    fi, ci, cols = _kept(L, W)
    Wm = (W.double().reshape(s.f, s.k) * _mask(L, fi, cols)).reshape(W.shape)
    b = torch.zeros(s.f, dtype=torch.float64, device=W.device)
    b[fi] = bias.double()[fi]
    ys = []
    step = max(1, int(2.5e8 // (s.c * s.t * s.h * s.w + s.f * s.plane)))
    for n0 in range(0, s.n, step):
        y = _conv64(s, x[n0:n0 + step].double(), Wm) + b.reshape((1, -1) + (1,) * (x.dim() - 2))
        ys.append(torch.relu(y) if relu else y)
    return fi, ci, torch.cat(ys)


def exact(case, seed):
    if case["op"] == "fwd":
        L, W, bias, x, _, _ = _layer_inputs(case, seed)
        return _fwd64(L, W, bias, x, case["relu"])[2]
    if case["op"] == "bwd":
        L, W, bias, x, dy, y = _layer_inputs(case, seed)
        s = L.shape
        fi, _, cols = _kept(L, W)
        mask = _mask(L, fi, cols)
        keep_f = torch.zeros(s.f, dtype=torch.float64, device=W.device)
        keep_f[fi] = 1.0
        Wm = (W.double().reshape(s.f, s.k) * mask).reshape(W.shape).requires_grad_(True)
        dW = torch.zeros(s.f, s.k, dtype=torch.float64, device=W.device)
        db = torch.zeros(s.f, dtype=torch.float64, device=W.device)
        dxs = []
        step = max(1, int(1.2e8 // (s.c * s.t * s.h * s.w + s.f * s.plane)))
        for n0 in range(0, s.n, step):
            dz = dy[n0:n0 + step].double() * keep_f.reshape((1, -1) + (1,) * (x.dim() - 2))
            if case["relu"]:
                dz = dz * (y[n0:n0 + step] > 0)
            xd = x[n0:n0 + step].double().requires_grad_(True)
            gx, gw = torch.autograd.grad(_conv64(s, xd, Wm), (xd, Wm), dz)
            dW += gw.reshape(s.f, s.k)
            db += dz.sum(dim=[0] + list(range(2, dz.dim())))
            dxs.append(gx)
        out = {"dW": dW * mask, "db": db}
        if case["dx"]:
            out["dx"] = torch.cat(dxs)
        return out
    if case["op"] == "admm":
        Ws, Us = _admm_inputs(case, seed)
        out = {"Z": [], "U": [], "filt": [], "cols": []}
        for L, W, U in zip(_net(case), Ws, Us):
            V = (W.double() + U.double()).to(W.dtype)  # one rounding to the tensors' precision
            fi, ci, cols = _kept(L, V)
            Z = (V.double().reshape(L.shape.f, L.shape.k) * _mask(L, fi, cols)).reshape(V.shape)
            out["Z"].append(Z)
            out["U"].append(V.double() - Z)
            out["filt"].append(fi)
            out["cols"].append(ci)
        return out
    out = {"filt": [], "cols": [], "y": []}
    for L, W, bias, x in _net_inputs(case, seed):
        fi, ci, y = _fwd64(L, W, bias, x, True)
        out["filt"].append(fi)
        out["cols"].append(ci)
        out["y"].append(y)
    return out
