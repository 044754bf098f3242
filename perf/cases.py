"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the public binding (``srn.py``, ``autograd.py``).
Inputs are made from a seed alone; ``exact`` restates each case in plain
64-bit torch, without the library.

Kinds of case
  eval    network output at scattered points (random-access decode)
  normals density and input gradient at scattered points
  train   one training pass through torch.autograd: forward, parameter and
          position gradients
  render  direct volume rendering of the network (the paper's main path)
  dense   direct volume rendering of the dense volume (the reference images)
  fit     optimiser steps of the fused fit, in the middle of a training
  error   the error grid that adaptive resampling refreshes
"""
import math

import numpy as np
import torch

from paper_2112_01579_gb300 import autograd, srn

#: Network shapes: latent grid vertices, channels, Fourier rows, layers, width, outputs, activation (0 sine, 1 SnakeAlt).
NETS = {
    "plain": dict(R=8, F=8, m=12, layers=2, width=32, D=1, act=0),     # the plain workload and its fit
    "main": dict(R=32, F=16, m=14, layers=4, width=32, D=1, act=1),    # the paper's main configuration
    "fine": dict(R=64, F=16, m=14, layers=4, width=32, D=1, act=1),    # the shaded workload
    "head": dict(R=32, F=16, m=14, layers=4, width=32, D=4, act=1),    # density and gradient outputs
    "small": dict(R=16, F=16, m=14, layers=2, width=32, D=1, act=1),   # the width / layer sweep, smallest
    "deep": dict(R=32, F=16, m=14, layers=6, width=32, D=1, act=1),    # the sweep at width 32, six layers
    "wide48": dict(R=32, F=16, m=22, layers=6, width=48, D=1, act=1),  # the paper's performance figure
    "wide64": dict(R=32, F=16, m=30, layers=4, width=64, D=1, act=1),
}
SHADING = {"none": srn.SRN_SHADE_NONE, "adjoint": srn.SRN_SHADE_ADJOINT, "fd": srn.SRN_SHADE_FD, "head": srn.SRN_SHADE_HEAD}


def listed():
    return [
        # a probe of a few values of a loaded network (picking, a profile line): latency and launches only
        dict(name="eval_probe", kind="eval", net="main", prec="fp16", n=1000, keys=1, u8=False),
        # the paper's random-access test, 10^6 locations
        dict(name="eval_decode", kind="eval", net="main", prec="fp16", n=1 << 20, keys=1, u8=False),
        # training with a torch optimiser: one ragged batch, forward and every gradient, FP32
        dict(name="train_batch", kind="train", net="main", n=65537, keys=1),
        # the plain FP32 workload: a thumbnail of the two-layer sine network
        dict(name="render_plain", kind="render", net="plain", prec="fp32", w=128, h=128, views=1, times=1, keys=1, u8=False,
             shading="none", inv_step=128, et=0.99),
        # the headline: one 1024^2 frame of the main configuration
        dict(name="render_main", kind="render", net="main", prec="fp16", w=1024, h=1024, views=1, times=1, keys=1, u8=False,
             shading="none", inv_step=512, et=0.99),
        # time-varying data: keyframes, several times and views in one call, odd image size
        dict(name="render_times", kind="render", net="main", prec="fp16", w=517, h=333, views=2, times=2, keys=5, u8=False,
             shading="none", inv_step=512, et=0.99),
        # shaded render with the adjoint gradient, the fine grid
        dict(name="render_shaded", kind="render", net="fine", prec="fp16", w=512, h=512, views=1, times=1, keys=1, u8=False,
             shading="adjoint", inv_step=1024, et=0.99),
        # the paper's performance figure: six layers of 48 channels, 512^2, no early termination
        dict(name="render_wide", kind="render", net="wide48", prec="fp16", w=512, h=512, views=1, times=1, keys=1, u8=False,
             shading="none", inv_step=256, et=2.0),
        # the reference image every comparison needs: the dense 256^3 volume at 1024^2
        dict(name="dense_volume", kind="dense", nx=256, ny=256, nz=256, w=1024, h=1024, views=1, shading="none", inv_step=512,
             et=0.99),
        # fit of the plain network, several replayed steps per call
        dict(name="fit_plain", kind="fit", net="plain", prec="fp32", n=1 << 18, volume=256, steps=4, adaptive=False),
        # fit of the main configuration, one step per call (a new volume may come every step)
        dict(name="fit_main", kind="fit", net="main", prec="fp16", n=1 << 18, volume=256, steps=1, adaptive=False),
        # adaptive resampling: the error grid at the paper's resolution and count
        dict(name="error_grid", kind="error", net="main", res=128, spv=8, volume=256),
    ]


def _log(rng, lo, hi):
    """A whole number, spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "normals", "train", "render", "render", "dense", "fit", "fit", "error"])
    if kind == "eval":
        prec = rng.choice(["fp16", "fp16", "fp32"])
        u8 = prec == "fp16" and rng.random() < 0.25
        return dict(kind=kind, net="main" if u8 else rng.choice(sorted(NETS)), prec=prec, n=_log(rng, 100, 1 << 20),
                    keys=1 if u8 else rng.choice([1, 1, 3]), u8=u8)
    if kind == "normals":
        return dict(kind=kind, net=rng.choice(["plain", "main", "head", "wide64"]), prec=rng.choice(["fp16", "fp32"]),
                    n=_log(rng, 100, 1 << 18), keys=rng.choice([1, 3]))
    if kind == "train":
        return dict(kind=kind, net=rng.choice(["plain", "main", "head", "small", "deep"]), n=_log(rng, 100, 1 << 18),
                    keys=rng.choice([1, 1, 3]))
    if kind == "render":
        prec = rng.choice(["fp16", "fp16", "fp16", "fp32"])
        most = 1024 if prec == "fp16" else 256
        net = rng.choice(["plain", "main", "fine", "head", "small", "wide48", "wide64"])
        shading = rng.choice(["none", "none", "adjoint", "fd"])
        if net == "head":
            shading = rng.choice(["none", "head"])
        if net == "wide48" and shading == "adjoint":
            shading = "none"  # six layers: deeper than the FP16 adjoint takes
        if shading == "fd":
            most = most // 4
        elif shading == "adjoint" or net.startswith("wide"):
            most = most // 2
        u8 = net == "main" and shading == "none" and prec == "fp16" and rng.random() < 0.25
        w, h = _log(rng, 16, most), _log(rng, 16, most)
        large = 4 * w * h > most * most
        return dict(kind=kind, net=net, prec=prec, w=w, h=h, views=1 if large else rng.choice([1, 2]), times=1,
                    keys=1 if u8 else rng.choice([1, 1, 3]), u8=u8, shading=shading, inv_step=rng.choice([128, 256, 512]),
                    et=0.99 if large else rng.choice([0.99, 2.0]))
    if kind == "dense":
        return dict(kind=kind, nx=_log(rng, 24, 320), ny=_log(rng, 24, 320), nz=_log(rng, 24, 320), w=_log(rng, 16, 1024),
                    h=_log(rng, 16, 1024), views=rng.choice([1, 2]), shading=rng.choice(["none", "fd"]),
                    inv_step=rng.choice([128, 256, 512]), et=rng.choice([0.99, 2.0]))
    if kind == "fit":
        net = rng.choice(["plain", "main", "small", "head"])
        return dict(kind=kind, net=net, prec="fp32" if net == "plain" else "fp16", n=_log(rng, 200, 1 << 18),
                    volume=_log(rng, 32, 256), steps=rng.choice([1, 2]), adaptive=rng.random() < 0.25)
    return dict(kind=kind, net=rng.choice(["plain", "main", "small", "wide48"]), res=_log(rng, 16, 96), spv=rng.choice([1, 4, 8]),
                volume=_log(rng, 32, 256))


# ------------------------------------------------------------------ inputs
def _rng(seed, salt):
    return np.random.default_rng([int(seed), salt])


def _network(case, seed):
    """Parameters of a trained-like network: Xavier weights, a latent grid of unit-order values, densities around 0.4.
    Values are FP16-representable, so the FP16 path's copies hold the same numbers."""
    s, rng = NETS[case["net"]], _rng(seed, 1)
    half = lambda a: np.asarray(a, np.float16).astype(np.float32)  # noqa: E731
    dims = [3 + 2 * s["m"] + s["F"]] + [s["width"]] * (s["layers"] - 1) + [s["D"]]
    W, b = [], []
    for din, dout in zip(dims[:-1], dims[1:]):
        a = math.sqrt(6.0 / (din + dout))
        W.append(half(rng.uniform(-a, a, (dout, din))))
        b.append(half(rng.normal(0.0, 0.1, dout)))
    W[-1] = half(0.35 * W[-1])
    W[-1][0] -= half(W[-1][0].mean())  # SnakeAlt activations have a mean of their own
    W[-1] = half(W[-1])
    b[-1][0] = half(0.4)
    keys = case.get("keys", 1)
    grid = rng.standard_normal((keys, s["R"], s["R"], s["R"], s["F"]), dtype=np.float32) * 0.3
    fourier = np.zeros((s["m"], 3), np.float32)
    for k in range(s["m"]):
        fourier[k, k % 3] = 2.0 * math.pi * 2.0 ** (k // 3)
    return dict(grid=half(grid), fourier=fourier, weights=W, biases=b, act=s["act"], key_times=4.0 * np.arange(keys, dtype=np.float32))


def _time(case):
    """The time a keyframed network is asked for: between two keyframes."""
    return 2.5 if case.get("keys", 1) > 1 else 0.0


def _times(case):
    return [1.5 + 3.0 * k for k in range(case["times"])] if case["keys"] > 1 else None


def _points(case, seed):
    return torch.from_numpy(_rng(seed, 2).random((case["n"], 3), dtype=np.float32)).cuda()


def _volume(nx, ny, nz, seed):
    """A density volume in [0, 1] with structure at several scales (float32 [nz, ny, nx])."""
    rng, v = _rng(seed, 3), torch.zeros((nz, ny, nx), device="cuda")
    for o, n in enumerate((5, 9, 17, 33, 65)):
        c = torch.from_numpy(rng.random((1, 1, n, n, n), dtype=np.float32)).cuda()
        v += 0.6 ** o * torch.nn.functional.interpolate(c, size=(nz, ny, nx), mode="trilinear", align_corners=True)[0, 0]
    v -= v.min()
    return (v / v.max()).contiguous()


def _cameras(case, seed):
    """Views from the unit sphere towards the middle of the volume."""
    az0, el = _rng(seed, 4).uniform(0.0, 2.0 * math.pi), math.radians(20.0)
    cams = []
    for k in range(case["views"]):
        az = az0 + 2.0 * math.pi * k / case["views"]
        eye = [math.cos(el) * math.cos(az), math.sin(el), math.cos(el) * math.sin(az)]
        cams.append(dict(eye=eye, target=[0.0, 0.0, 0.0], up=[0.0, 1.0, 0.0], fovy=math.radians(90.0)))
    return cams


def _tf(case):
    """The four- and eight-point transfer functions of the workloads."""
    if case.get("net") == "plain":
        pos = [0.0, 0.35, 0.65, 1.0]
        rgba = [[0.0, 0.0, 0.0, 0.0], [0.2, 0.4, 1.0, 0.05], [1.0, 0.6, 0.2, 0.4], [1.0, 1.0, 1.0, 1.0]]
    else:
        pos = [0.0, 0.2, 0.3, 0.4, 0.55, 0.7, 0.85, 1.0]
        rgba = [[0.0, 0.0, 0.0, 0.0], [0.1, 0.2, 0.9, 0.0], [0.2, 0.5, 1.0, 0.15], [0.3, 0.9, 0.6, 0.02],
                [0.9, 0.9, 0.2, 0.3], [1.0, 0.5, 0.1, 0.05], [1.0, 0.2, 0.1, 0.6], [1.0, 1.0, 1.0, 1.0]]
    return dict(pos=np.asarray(pos, np.float32), rgba=np.asarray(rgba, np.float32), opacity_scale=20.0)


def _moments(case, seed, p):
    """Adam moments as a training some hundred steps old has them: each entry's gradient scale from the points that reach
    it, the first moment a part of it."""
    s, rng, n = NETS[case["net"]], _rng(seed, 5), case["n"]
    cells = (s["R"] - 1) ** 3
    scale = np.concatenate([np.full(p["grid"].size, 0.3 / n * math.sqrt(n / cells / 3.4 + 0.1), np.float32),
                            np.full(sum(w.size for w in p["weights"]) + sum(b.size for b in p["biases"]), 0.5 / math.sqrt(n), np.float32)])
    v = (scale * (0.5 + rng.random(scale.size, dtype=np.float32))) ** 2
    m = 0.3 * scale * rng.standard_normal(scale.size, dtype=np.float32)
    return m.astype(np.float32), v.astype(np.float32)


STEP0 = 500  # the training step a fit case starts at
LR_GRID, LR_NET = 1e-2, 5e-3
GRAD_WEIGHT, GRAD_SCALE = 0.01, 0.05  # of the gradient head's loss


def _error_grid_input(case, seed):
    """A past error grid, 32^3: a few regions carry most of the error."""
    return torch.from_numpy((_rng(seed, 6).random((32, 32, 32), dtype=np.float32) ** 4 * 0.1).astype(np.float32)).cuda()


# ------------------------------------------------------------------ prepare / run
def prepare(case, seed):
    kind, s = case["kind"], dict(case=case)
    prec = srn.SRN_PREC_FP32 if case.get("prec", "fp32") == "fp32" else srn.SRN_PREC_FP16
    if kind == "dense":
        s["volume"] = _volume(case["nx"], case["ny"], case["nz"], seed)
    else:
        p = _network(case, seed)
    if kind == "train":
        s["module"] = autograd.SRNModule(p, max_batch=case["n"])
        s["pts"] = _points(case, seed).requires_grad_(True)
        s["dout"] = torch.from_numpy(_rng(seed, 7).standard_normal((case["n"], NETS[case["net"]]["D"]), dtype=np.float32)).cuda()
        return s
    if kind == "fit":
        s["net"] = srn.Network(p, precision=prec, max_fit_points=case["n"], adam=True)
        m, v = _moments(case, seed, p)
        s["net"].adam_m.copy_(torch.from_numpy(m))
        s["net"].adam_v.copy_(torch.from_numpy(v))
        s["volume"] = _volume(case["volume"], case["volume"], case["volume"], seed)
        s["loss"], s["step"] = torch.zeros(1, device="cuda"), STEP0
        if case["adaptive"]:
            srn.srn_fit_set_sampling(s["net"].ctx, _error_grid_input(case, seed), 32)
        return s
    if kind != "dense":
        s["net"] = srn.Network(p, precision=prec, grid_u8=case.get("u8", False))
    if kind in ("eval", "normals"):
        s["pts"], D = _points(case, seed), NETS[case["net"]]["D"]
        s["out"] = torch.empty((case["n"], D) if kind == "eval" else case["n"], device="cuda")
        s["grad"] = torch.empty((case["n"], 3), device="cuda")
    elif kind == "error":
        s["volume"] = _volume(case["volume"], case["volume"], case["volume"], seed)
        s["err"] = torch.empty(case["res"] ** 3, device="cuda")
    else:
        s["cams"], s["tf"] = _cameras(case, seed), _tf(case)
        s["desc"] = srn.render_desc(case["w"], case["h"], 1.0 / case["inv_step"], case["et"], SHADING[case["shading"]], _fd_h(case))
        s["image"] = torch.empty((case.get("times", 1), case["views"], case["h"], case["w"], 4), device="cuda")
    return s


def _fd_h(case):
    return 1.0 / 255.0 if case["shading"] == "fd" else 0.0


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "eval":
        srn.srn_eval(s["net"].ctx, s["pts"], s["out"], time=_time(case))
        return s["out"]
    if kind == "normals":
        srn.srn_density_grad(s["net"].ctx, s["pts"], s["out"], s["grad"], time=_time(case))
        return s["out"], s["grad"]
    if kind == "train":
        m, pts = s["module"], s["pts"]
        pts.grad = m.grid.grad = m.weights.grad = m.biases.grad = None
        out = m(pts, _time(case))
        out.backward(s["dout"])
        return dict(out=out.detach(), pts=pts.grad, grid=m.grid.grad, weights=m.weights.grad, biases=m.biases.grad)
    if kind == "render":
        srn.srn_render(s["net"].ctx, s["cams"], s["tf"], s["desc"], s["image"], times=_times(case))
        return s["image"]
    if kind == "dense":
        srn.srn_dvr_dense(s["volume"], s["cams"], s["tf"], s["desc"], s["image"])
        return s["image"]
    net = s["net"]
    if kind == "error":
        srn.srn_error_grid(net.ctx, s["volume"], case["res"], case["spv"], 17, s["err"])
        return s["err"]
    args = dict(lr_grid=LR_GRID, lr_net=LR_NET, grad_weight=GRAD_WEIGHT if net.out_dim == 4 else 0.0, grad_scale=GRAD_SCALE)
    if case["steps"] == 1:
        srn.srn_fit_step(net.ctx, s["volume"], case["n"], 23, s["step"], s["loss"], **args)
    else:
        srn.srn_fit_steps(net.ctx, s["volume"], case["n"], 23, s["step"], case["steps"], s["loss"], **args)
    s["step"] += case["steps"]
    return dict(grid=net.grid, weights=net.weights, biases=net.biases, m=net.adam_m, v=net.adam_v, loss=s["loss"])


# ------------------------------------------------------------------ work
def _net_flops(case):
    s = NETS[case["net"]]
    dims = [3 + 2 * s["m"] + s["F"]] + [s["width"]] * (s["layers"] - 1) + [s["D"]]
    return 2 * sum(a * b for a, b in zip(dims[:-1], dims[1:])) + 16 * s["F"]


def _net_bytes(case, each=4):
    s = NETS[case["net"]]
    dims = [3 + 2 * s["m"] + s["F"]] + [s["width"]] * (s["layers"] - 1) + [s["D"]]
    return each * (case.get("keys", 1) * s["R"] ** 3 * s["F"] + sum(a * b + b for a, b in zip(dims[:-1], dims[1:])))


def work(case):
    """One pass: every input read and every output written once, the network's multiply-adds and the trilinear blends."""
    kind = case["kind"]
    each = 1 if case.get("u8") else (2 if case.get("prec") == "fp16" else 4)
    if kind in ("eval", "normals"):
        outs = 4 if kind == "normals" else NETS[case["net"]]["D"]
        return dict(bytes=case["n"] * 4 * (3 + outs) + _net_bytes(case, each), flops=case["n"] * _net_flops(case) * (2 if kind == "normals" else 1))
    if kind == "train":
        return dict(bytes=case["n"] * 4 * (3 + 3 + 2 * NETS[case["net"]]["D"]) + 2 * _net_bytes(case), flops=3 * case["n"] * _net_flops(case))
    if kind == "fit":
        return dict(bytes=case["steps"] * (7 * _net_bytes(case) + 4 * min(case["volume"] ** 3, 8 * case["n"])), flops=3 * case["steps"] * case["n"] * _net_flops(case))
    if kind == "error":
        return dict(bytes=4 * (case["res"] ** 3 + case["volume"] ** 3) + _net_bytes(case), flops=case["res"] ** 3 * case["spv"] * _net_flops(case))
    samples = _samples(case)
    image = 16 * case.get("times", 1) * case["views"] * case["w"] * case["h"]
    if kind == "dense":
        return dict(bytes=image + 4 * case["nx"] * case["ny"] * case["nz"], flops=samples * 15 * (7 if case["shading"] == "fd" else 1))
    passes = {"none": 1, "head": 1, "adjoint": 2, "fd": 7}[case["shading"]]
    return dict(bytes=image + _net_bytes(case, each), flops=samples * passes * _net_flops(case))


def _samples(case):
    """Samples of a pass, from every 64th pixel (seed 0's scene) with the early termination it has."""
    total = 0
    for _, march in _marches(case, 0, stride=8):
        total += march(count_only=True)
    return 64 * total


# ------------------------------------------------------------------ exact
class _Net64:
    def __init__(self, case, p):
        t = lambda a: torch.from_numpy(np.asarray(a)).cuda().double()  # noqa: E731
        self.grid, self.fourier, self.act = t(p["grid"]), t(p["fourier"]), p["act"]
        if case.get("u8"):  # per channel: codes 0..255 over [min, max], found in 32 bits as the interface states
            g = torch.from_numpy(p["grid"]).cuda()
            F = g.shape[-1]
            lo, hi = g.reshape(-1, F).amin(0), g.reshape(-1, F).amax(0)
            step = torch.where(hi > lo, (hi - lo) / 255.0, torch.ones_like(lo))
            self.grid = lo.double() + step.double() * torch.round((g - lo) / step).clamp(0, 255).double()
        self.W, self.b = [t(w) for w in p["weights"]], [t(b) for b in p["biases"]]
        self.key_times = [float(k) for k in p["key_times"]]

    def blended(self, time):
        """The latent grid at one time, [R^3, F]."""
        g, kt = self.grid, self.key_times
        F = g.shape[-1]
        if g.shape[0] == 1:
            return g[0].reshape(-1, F)
        time = float(np.float32(time))
        k = 0
        while k < len(kt) - 2 and time >= kt[k + 1]:
            k += 1
        f = min(max((time - kt[k]) / (kt[k + 1] - kt[k]), 0.0), 1.0)
        return ((1.0 - f) * g[k] + f * g[k + 1]).reshape(-1, F)

    def __call__(self, pts, grid, W=None, b=None):
        R, W, b = self.grid.shape[1], W or self.W, b or self.b
        e = pts @ self.fourier.T
        z = _trilinear(grid, pts, (R, R, R))
        x = torch.cat([pts, torch.sin(e), torch.cos(e), z], 1)
        for i, (w, c) in enumerate(zip(W, b)):
            x = torch.addmm(c, x, w.T)
            if i < len(W) - 1:
                x = 0.5 * x + torch.sin(x) ** 2 if self.act else torch.sin(x)
        return x


def _trilinear(values, pts, dims):
    """values [nz * ny * nx, F] with x fastest, vertex aligned, at pts in [0, 1]^3."""
    i, f = [], []
    for a in range(3):
        g = pts[:, a] * (dims[a] - 1)
        k = g.detach().floor().clamp(0, dims[a] - 2)
        i.append(k.long())
        f.append(g - k)
    out = 0
    for c in range(8):
        w, at = 1, 0
        for a, stride in zip(range(3), (1, dims[0], dims[0] * dims[1])):
            d = (c >> a) & 1
            w = w * (f[a] if d else 1 - f[a])
            at = at + (i[a] + d) * stride
        out = out + w[:, None] * values[at]
    return out


def _colour(tf, rho):
    pos, rgba = torch.from_numpy(tf["pos"]).cuda().double(), torch.from_numpy(tf["rgba"]).cuda().double()
    x = rho.clamp(0, 1)
    i = (torch.searchsorted(pos, x.contiguous(), right=True) - 1).clamp(0, len(pos) - 2)
    f = ((x - pos[i]) / (pos[i + 1] - pos[i])).clamp(0, 1)[:, None]
    return (1 - f) * rgba[i] + f * rgba[i + 1]


def _field(case, seed, time):
    """A function of points [n, 3]: density and, where the case shades, its gradient."""
    if case["kind"] == "dense":
        dims = (case["nx"], case["ny"], case["nz"])
        v = _volume(*dims, seed).double().reshape(-1, 1)
        rho, h = (lambda p: _trilinear(v, p, dims)[:, 0]), [1.0 / (n - 1) for n in dims]
    else:
        net = _Net64(case, _network(case, seed))
        g = net.blended(time)
        rho, h = (lambda p: net(p, g)[:, 0]), [float(np.float32(_fd_h(case)))] * 3

    def central(p):
        out = []
        for a in range(3):
            d = torch.zeros(3, device="cuda", dtype=torch.float64)
            d[a] = h[a]
            out.append((rho((p + d).clamp(0, 1)) - rho((p - d).clamp(0, 1))) / (2 * h[a]))
        return torch.stack(out, 1)

    def field(p):
        if case["shading"] == "none":
            return rho(p), None
        if case["shading"] == "fd":
            return rho(p), central(p)
        if case["shading"] == "head":
            o = net(p, g)
            return o[:, 0], o[:, 1:4]
        with torch.enable_grad():
            q = p.clone().requires_grad_(True)
            r = rho(q)
            grad, = torch.autograd.grad(r.sum(), q)
        return r.detach(), grad
    return field


def _marches(case, seed, stride=1):
    """(frame, march) for every time and view; march() gives the frame's pixels [n, 4], or its number of samples."""
    f32 = lambda v: float(np.float32(v))  # noqa: E731
    step, et, tf, shaded = f32(1.0 / case["inv_step"]), f32(case["et"]), _tf(case), case["shading"] != "none"
    times = _times(case) if case["kind"] == "render" and case["keys"] > 1 else [0.0] * case.get("times", 1)
    for t, time in enumerate(times):
        field = _field(case, seed, time)
        for c, cam in enumerate(_cameras(case, seed)):
            v3 = lambda a: torch.tensor([f32(x) for x in a], dtype=torch.float64, device="cuda")  # noqa: E731
            eye, target, up, th = v3(cam["eye"]), v3(cam["target"]), v3(cam["up"]), math.tan(0.5 * f32(cam["fovy"]))
            fw = (target - eye) / (target - eye).norm()
            right = torch.linalg.cross(fw, up)
            right = right / right.norm()
            upv = torch.linalg.cross(right, fw)
            W, H = case["w"], case["h"]
            x = torch.arange(min(stride // 2, W - 1), W, stride, device="cuda", dtype=torch.float64)
            y = torch.arange(min(stride // 2, H - 1), H, stride, device="cuda", dtype=torch.float64)
            sx, sy = (2 * (x + 0.5) / W - 1) * th * (W / H), (1 - 2 * (y + 0.5) / H) * th
            d = (fw + sx[None, :, None] * right + sy[:, None, None] * upv).reshape(-1, 3)
            d = d / d.norm(dim=1, keepdim=True)
            ta, tb = (-0.5 - eye) / d, (0.5 - eye) / d
            t0, t1 = torch.minimum(ta, tb).amax(1).clamp_min(0), torch.maximum(ta, tb).amin(1)

            @torch.no_grad()
            def march(count_only=False):
                out = torch.zeros((len(d), 4), device="cuda", dtype=torch.float64)
                live, k, samples = torch.nonzero(t1 > t0)[:, 0], 0, 0
                while len(live):
                    samples += len(live)
                    a = t0[live] + k * step
                    b = torch.minimum(t0[live] + (k + 1) * step, t1[live])
                    rgba = torch.empty((len(live), 4), device="cuda", dtype=torch.float64)
                    for part in torch.arange(len(live), device="cuda").split(1 << 18):
                        p = (eye + (0.5 * (a[part] + b[part]))[:, None] * d[live[part]] + 0.5).clamp(0, 1)
                        rho, grad = field(p)
                        col = _colour(tf, rho)
                        if shaded:
                            norm = grad.norm(dim=1)
                            cosine = (grad * d[live[part]]).sum(1).abs() / norm.clamp_min(1e-30)
                            lit = col[:, :3] * (0.1 + 0.6 * cosine)[:, None] + 0.3 * (cosine ** 32)[:, None]
                            col = torch.cat([torch.where((norm >= 1e-6)[:, None], lit, col[:, :3]), col[:, 3:]], 1)
                        rgba[part] = col
                    alpha = 1 - torch.exp(-rgba[:, 3] * tf["opacity_scale"] * (b - a))
                    w = (1 - out[live, 3]) * alpha
                    out[live] += torch.cat([w[:, None] * rgba[:, :3], w[:, None]], 1)
                    k += 1
                    live = live[(out[live, 3] < et) & (t0[live] + k * step < t1[live])]
                return samples if count_only else out
            yield (t, c), march


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 of counters (int64 tensors holding 32-bit words)."""
    m = 0xFFFFFFFF

    def product(a, mul):  # high and low words of a 32 x 32 bit product
        lo, hi = (a & 0xFFFF) * mul, (a >> 16) * mul
        return ((hi + (lo >> 16)) >> 16) & m, (lo + ((hi & 0xFFFF) << 16)) & m
    for r in range(10):
        h0, l0 = product(c0, 0xD2511F53)
        h1, l1 = product(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1, c2


def _drawn_points(case, seed, step):
    """The points of one fit step: uniform, or in proportion to the past error grid."""
    j = torch.arange(case["n"], device="cuda")
    zero = torch.zeros_like(j)
    u = [((w >> 8).float() * 2.0 ** -24) for w in _philox(j, zero + step, zero + 0x5352, zero, zero + 23, zero)]
    if not case["adaptive"]:
        return torch.stack(u, 1)
    E, n = _error_grid_input(case, seed).reshape(-1), case["n"]
    q = torch.floor(E * (torch.tensor(65535.0, device="cuda") / E.max())).clamp(max=65535.0).long()
    S = torch.cat([q.new_zeros(1), torch.cumsum(q, 0)])
    v = torch.searchsorted(S, ((2 * j + 1) * S[-1]) // (2 * n), right=True) - 1
    return torch.stack([((c.float() + w) / 32.0) for c, w in zip((v % 32, v // 32 % 32, v // 1024), u)], 1)


def _exact_fit(case, seed):
    p, s = _network(case, seed), NETS[case["net"]]
    net, nv, n = _Net64(case, p), case["volume"], case["n"]
    vol = _volume(nv, nv, nv, seed).double().reshape(-1, 1)
    m, v = (torch.from_numpy(a).cuda().double() for a in _moments(case, seed, p))
    grid = net.grid[0].reshape(-1, s["F"])
    params = [grid] + net.W + net.b
    lr = [float(np.float32(LR_GRID))] + [float(np.float32(LR_NET))] * (len(params) - 1)
    gw, gs = float(np.float32(GRAD_WEIGHT)), float(np.float32(GRAD_SCALE))
    for k in range(case["steps"]):
        step = STEP0 + k
        pts, loss = _drawn_points(case, seed, step).double(), 0.0
        params = [q.detach().requires_grad_(True) for q in params]
        total = [torch.zeros_like(q) for q in params]
        for part in pts.split(1 << 16):
            out = net(part, params[0], params[1:1 + s["layers"]], params[1 + s["layers"]:])
            l = (out[:, 0] - _trilinear(vol, part, (nv, nv, nv))[:, 0]).abs().sum()
            if s["D"] == 4:
                h = float(np.float32(1.0) / np.float32(nv - 1))
                for a in range(3):
                    d = torch.zeros(3, device="cuda", dtype=torch.float64)
                    d[a] = h
                    g = (_trilinear(vol, (part + d).clamp(0, 1), (nv,) * 3) - _trilinear(vol, (part - d).clamp(0, 1), (nv,) * 3))[:, 0] / (2 * h)
                    l = l + gw * (out[:, 1 + a] - gs * g).abs().sum()
            l = l / n
            for t, g in zip(total, torch.autograd.grad(l, params)):
                t += g
            loss += float(l.detach())
        g = torch.cat([t.reshape(-1) for t in total])
        b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
        m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
        up = (m / (1 - b1 ** (step + 1))) / (torch.sqrt(v / (1 - b2 ** (step + 1))) + 1e-8)
        ups = up.split([q.numel() for q in params])
        params = [q.detach() - r * u.reshape(q.shape) for q, r, u in zip(params, lr, ups)]
    flat = lambda ts: torch.cat([q.reshape(-1) for q in ts])  # noqa: E731
    return dict(grid=params[0].reshape(-1), weights=flat(params[1:1 + s["layers"]]), biases=flat(params[1 + s["layers"]:]), m=m, v=v,
                loss=torch.tensor([loss], dtype=torch.float64))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("render", "dense"):
        out = torch.zeros((case.get("times", 1), case["views"], case["h"], case["w"], 4), device="cuda", dtype=torch.float64)
        for (t, c), march in _marches(case, seed):
            out[t, c] = march().reshape(case["h"], case["w"], 4)
        return out
    if kind == "fit":
        return _exact_fit(case, seed)
    net = _Net64(case, _network(case, seed))
    grid = net.blended(_time(case))
    if kind == "error":
        res, n = case["res"], case["volume"]
        vol = _volume(n, n, n, seed).double().reshape(-1, 1)
        v = torch.arange(res ** 3, device="cuda")
        zero, err = torch.zeros_like(v), torch.zeros(res ** 3, device="cuda", dtype=torch.float64)
        for i in range(case["spv"]):
            u = _philox(v, zero + i, zero + 0x4552, zero, zero + 17, zero)
            p = torch.stack([(c.float() + (w >> 8).float() * 2.0 ** -24) / np.float32(res)
                             for c, w in zip((v % res, v // res % res, v // res ** 2), u)], 1).double()
            for part in v.split(1 << 18):
                err[part] += (net(p[part], grid)[:, 0] - _trilinear(vol, p[part], (n, n, n))[:, 0]).abs()
        return err / case["spv"]
    pts = _points(case, seed).double()
    if kind == "eval":
        return torch.cat([net(p, grid) for p in pts.split(1 << 18)])
    if kind == "normals":
        rho, grad = [], []
        for p in pts.split(1 << 16):
            p = p.clone().requires_grad_(True)
            r = net(p, grid)[:, 0]
            grad.append(torch.autograd.grad(r.sum(), p)[0])
            rho.append(r.detach())
        return torch.cat(rho), torch.cat(grad)
    dout = torch.from_numpy(_rng(seed, 7).standard_normal((case["n"], NETS[case["net"]]["D"]), dtype=np.float32)).cuda().double()
    g = net.grid.clone().requires_grad_(True)
    net.grid = g
    W, b = [w.requires_grad_(True) for w in net.W], [c.requires_grad_(True) for c in net.b]
    out, dp = [], []
    total = [torch.zeros_like(q) for q in [g] + W + b]
    for p, do in zip(pts.split(1 << 16), dout.split(1 << 16)):
        p = p.clone().requires_grad_(True)
        o = net(p, net.blended(_time(case)))
        grads = torch.autograd.grad((o * do).sum(), [p, g] + W + b)
        out.append(o.detach())
        dp.append(grads[0])
        for t, q in zip(total, grads[1:]):
            t += q
    flat = lambda ts: torch.cat([q.reshape(-1) for q in ts])  # noqa: E731
    return dict(out=torch.cat(out), pts=torch.cat(dp), grid=total[0].reshape(-1), weights=flat(total[1:1 + len(W)]), biases=flat(total[1 + len(W):]))
