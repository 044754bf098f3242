"""The FP32 tile kernels (32 points per warp) at the sizes where a tile, a
CTA or a row block ends: point counts around 32 and 128, every input-row
remainder, two to eight layers, general Fourier matrices and arguments beyond
the inline sine's range, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2112_01579_gb300 import synth

pytestmark = pytest.mark.gpu

# Largest gradient entry's share an entry may be off: the bound of the other
# FP32 gradient tests (sums of at most 10^3 FP32 products).
TOL_GRAD = 2e-5


@pytest.fixture(scope="module")
def S():
    from paper_2112_01579_gb300 import build
    build.build()
    from paper_2112_01579_gb300 import srn
    return srn


def _rel(a, b):
    a, b = np.asarray(a, np.float64).ravel(), np.asarray(b, np.float64).ravel()
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-30))


def _flat(parts):
    return np.concatenate([np.asarray(x).ravel() for x in parts])


# (layers, latent channels, Fourier rows, outputs, time input, keyframes): 48
# inputs is the most the tiled backward takes, five layers take the other one
BACKWARD = [(2, 8, 12, 1, 0, 1), (3, 4, 0, 4, 0, 1), (4, 16, 14, 1, 1, 3), (4, 16, 14, 4, 0, 1), (3, 32, 6, 1, 0, 1),
            (4, 16, 15, 1, 0, 1), (5, 16, 14, 1, 0, 1)]


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 1000])
@pytest.mark.parametrize("shape", BACKWARD)
def test_backward_matches_oracle(S, shape, n):
    import torch
    layers, F, m, D, ti, keys = shape
    p = synth.random_params(R=5, F=F, m=m, layers=layers, width=32, out_dim=D, act=synth.ACT_SNAKEALT, seed=n, grid_std=0.5,
                            n_keyframes=keys, time_input=ti)
    net = S.Network(p, max_fit_points=1000)
    rng = np.random.default_rng(n + 1)
    pts, dout = rng.random((n, 3), dtype=np.float32), rng.standard_normal((n, D), dtype=np.float32)
    g, w, b = (torch.full_like(t, float("nan")) for t in (net.grid, net.weights, net.biases))
    t = 0.75 if keys > 1 else 0.0
    S.srn_backward(net.ctx, torch.tensor(pts, device="cuda"), torch.tensor(dout, device="cuda"), g, w, b, time=t)
    rW, rb, rg = oracle.net_backward(oracle.OracleNet(p), pts, dout, t)
    assert _rel(g.cpu().numpy(), rg) <= TOL_GRAD
    assert _rel(w.cpu().numpy(), _flat(rW)) <= TOL_GRAD
    assert _rel(b.cpu().numpy(), _flat(rb)) <= TOL_GRAD


def _points(n, seed):
    pts = np.random.default_rng(seed).random((n, 3), dtype=np.float32)
    pts[0] = [1.0, 0.0, 0.5]
    return pts


@pytest.mark.parametrize("n", [1, 31, 33, 129, 2500])
@pytest.mark.parametrize("width,layers,m,nerf", [(32, 2, 12, True), (32, 8, 0, True), (32, 3, 33, True), (32, 4, 14, False),
                                                 (48, 3, 22, True), (64, 2, 30, True)])
def test_eval_matches_oracle(S, width, layers, m, nerf, n):
    """Densities to 1e-5 of max(|rho|, 1), the gradient to its first-order
    rounding-error bound, the one seeded with output adjoints to 1e-4 of
    max(|g|, 1): the FP32 bounds.  33 NeRF rows and a general matrix take the
    accurate library sine."""
    import torch
    p = synth.random_params(R=6, F=8, m=m, layers=layers, width=width, out_dim=4, act=synth.ACT_SNAKEALT, seed=n, grid_std=0.5)
    if not nerf:
        p["fourier"] = np.random.default_rng(5).normal(0, 8, (m, 3)).astype(np.float32)
    net, on, pts = S.Network(p), oracle.OracleNet(p), _points(n, n)
    x = torch.tensor(pts, device="cuda")
    out = torch.full((n, 4), float("nan"), device="cuda")
    S.srn_eval(net.ctx, x, out)
    ref = oracle.net_forward(on, pts)
    assert (np.abs(out.cpu().numpy() - ref) / np.maximum(np.abs(ref), 1.0)).max() <= 1e-5
    rho, grad = torch.full((n,), float("nan"), device="cuda"), torch.full((n, 3), float("nan"), device="cuda")
    S.srn_density_grad(net.ctx, x, rho, grad)
    rref, gref = oracle.net_input_grad(on, pts)
    assert torch.equal(rho, out[:, 0])
    assert (np.abs(grad.cpu().numpy() - gref) / oracle.error_bounds(on, pts, oracle.PREC_FP32)[1]).max() <= 1.0
    dout = np.random.default_rng(n + 9).standard_normal((n, 4), dtype=np.float32)
    S.srn_input_backward(net.ctx, x, torch.tensor(dout, device="cuda"), grad)
    vref = oracle.net_input_vjp(on, pts, dout)
    assert (np.abs(grad.cpu().numpy() - vref) / np.maximum(np.abs(vref).max(axis=1, keepdims=True), 1.0)).max() <= 1e-4


@pytest.mark.parametrize("act", [synth.ACT_SINE, synth.ACT_SNAKEALT])
@pytest.mark.parametrize("arg", [9999.0, 1.0e4, 10001.0, 3.0e7])
def test_eval_large_arguments(S, act, arg):
    """Pre-activations at both sides of the inline sine's range, exact in FP32
    (a bias alone), so only the sine's own error counts (1e-6, against weights
    of at most 1); SnakeAlt's linear part takes no weight."""
    import torch
    p = synth.random_params(R=4, F=4, m=3, layers=2, width=32, act=act, seed=3, grid_std=0.5)
    for k, sign in ((0, 1.0), (17, -1.0)):
        p["weights"][0][k] = 0.0
        p["biases"][0][k] = sign * arg
        if act == synth.ACT_SNAKEALT:
            p["weights"][1][0, k] = 0.0
    if act == synth.ACT_SINE:
        p["weights"][1][0, 0], p["weights"][1][0, 17] = 1.0, -0.5
    net, pts = S.Network(p), _points(33, 4)
    out = torch.full((33, 1), float("nan"), device="cuda")
    S.srn_eval(net.ctx, torch.tensor(pts, device="cuda"), out)
    ref = oracle.net_forward(oracle.OracleNet(p), pts)
    assert np.abs(out.cpu().numpy() - ref).max() <= 2e-6
    rho, grad = torch.empty(33, device="cuda"), torch.empty((33, 3), device="cuda")
    S.srn_density_grad(net.ctx, torch.tensor(pts, device="cuda"), rho, grad)
    gref = oracle.net_input_grad(oracle.OracleNet(p), pts)[1]
    assert (np.abs(grad.cpu().numpy() - gref) / np.maximum(np.abs(gref).max(axis=1, keepdims=True), 1.0)).max() <= 1e-4


@pytest.mark.parametrize("width,m,most", [(32, 14, 8), (48, 22, 6), (64, 30, 7)])
def test_fp16_depths(S, width, m, most):
    """The depths the FP16 path takes at each width, and the next one refused."""
    import torch
    for layers in {most, min(most + 1, 8)}:
        p = synth.to_half_exact(synth.random_params(R=3, F=16, m=m, layers=layers, width=width, act=synth.ACT_SNAKEALT, seed=layers))
        net, pts = S.Network(p, precision=S.SRN_PREC_FP16), _points(200, 1)
        out = torch.full((200, 1), float("nan"), device="cuda")
        if layers > most:
            with pytest.raises(S.SrnError) as e:
                S.srn_eval(net.ctx, torch.tensor(pts, device="cuda"), out)
            assert e.value.status == S.SRN_ERR_UNSUPPORTED
            continue
        S.srn_eval(net.ctx, torch.tensor(pts, device="cuda"), out)
        on = oracle.OracleNet(p)
        bound = oracle.error_bounds(on, pts, oracle.PREC_FP16, grad=False)[0]
        assert (np.abs(out.cpu().numpy() - oracle.net_forward(on, pts)) / bound).max() <= 1.0


@pytest.mark.parametrize("width,per_sm,extra", [(32, 4, 1), (32, 5, -31), (32, 13, 7), (32, 16, 0), (32, 16, 1), (64, 4, 33), (64, 8, 0)])
def test_calls_between_one_wave_and_many(S, width, per_sm, extra):
    """Point calls whose tiles give each SM one CTA of 4 to 16 warps (a tile
    each), at the edges of that range: the same bits as the points in calls of
    1000, each point being evaluated by itself."""
    import torch
    p = synth.random_params(R=5, F=16, m=14 if width == 32 else 30, layers=4, width=width, act=synth.ACT_SNAKEALT, seed=per_sm,
                            grid_std=0.5)
    n = 32 * per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    net = S.Network(p)
    pts = torch.tensor(_points(n, 6), device="cuda")
    dout = torch.randn((n, 1), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    whole, parts = ([torch.full(s, float("nan"), device="cuda") for s in ((n, 1), (n,), (n, 3), (n, 3))] for _ in range(2))
    for bufs, size in ((whole, n), (parts, 1000)):
        for i in range(0, n, size):
            out, rho, grad, vjp = (b[i : i + size] for b in bufs)
            S.srn_eval(net.ctx, pts[i : i + size], out)
            S.srn_density_grad(net.ctx, pts[i : i + size], rho, grad)
            S.srn_input_backward(net.ctx, pts[i : i + size], dout[i : i + size], vjp)
    for a, b in zip(whole, parts):
        assert torch.equal(a, b) and torch.isfinite(a).all()


# (width, layers, latent channels, Fourier rows, outputs, shading): more than 128 inputs, where a render's CTA takes all
# the shared memory an SM gives one but the transfer function's
WIDE_INPUT = [(64, 7, 32, 57, 4, 1), (64, 8, 8, 79, 4, 0), (64, 8, 32, 110, 1, 0), (32, 8, 4, 124, 1, 0)]


@pytest.mark.parametrize("width,layers,F,m,D,shading", WIDE_INPUT)
def test_render_of_wide_inputs(S, width, layers, F, m, D, shading):
    """The image against the oracle.  With the transfer function of slope 1
    and extinction 4 rho over rays of at most 1.74, a density error e moves a
    pixel by at most (2 4 1.74 + 1) e < 16 e; e is twice the largest FP32
    bound of 2000 points.  Shading adds its own bound."""
    import torch
    p = synth.random_params(R=4, F=F, m=m, layers=layers, width=width, out_dim=D, act=synth.ACT_SNAKEALT, seed=m, grid_std=0.5)
    p["fourier"] = np.random.default_rng(6).normal(0, 6, (m, 3)).astype(np.float32)
    net, on = S.Network(p), oracle.OracleNet(p)
    tf = dict(pos=np.asarray([0.0, 1.0], np.float32), rgba=np.asarray([[0, 0, 0, 0], [1, 1, 1, 1]], np.float32), opacity_scale=4.0)
    otf, cams = oracle.OracleTF(tf["pos"], tf["rgba"], 4.0), synth.orbit_cameras(1)
    out = torch.full((1, 1, 12, 17, 4), float("nan"), device="cuda")
    S.srn_render(net.ctx, cams, tf, S.render_desc(17, 12, 1 / 24, 2.0, shading), out)
    tol = 16 * 2 * float(oracle.error_bounds(on, _points(2000, 7), oracle.PREC_FP32, grad=False)[0].max())
    if shading:
        ref, bound = oracle.render_shade_bound(on, cams, otf, 17, 12, 1 / 24, 2.0, shading, oracle.PREC_FP32)
        err, lim = np.abs(out.cpu().numpy() - ref).max(axis=-1).ravel(), tol + np.asarray(bound).ravel()
    else:
        ref, _, _ = oracle.render(on, cams, otf, 17, 12, 1 / 24, 2.0)
        err, lim = np.abs(out.cpu().numpy() - ref).max(axis=-1).ravel(), tol
    assert tol < 1e-2 and (err <= lim).all(), (err.max(), tol)


@pytest.mark.parametrize("path", ["density_grad", "backward"])
@pytest.mark.parametrize("scale", [4.0, 64.0])
def test_sine_derivative_is_a_cosine_to_a_rounding(S, path, scale):
    """One sine neuron, arguments exact in FP32 (4913 vertices of a 17^3 grid
    spell multiples of 2^-10 times scale / 4), weights powers of two, one
    point per vertex: what comes back is the cosine alone.  Its rms error is
    at most 1.45 times that of the correctly rounded one (CUDA's own cosine:
    1.35; sin(pi / 2 - |r|) from a reduced r: 1.8)."""
    import torch
    p = synth.random_params(R=17, F=4, m=0, layers=2, width=32, act=synth.ACT_SINE, seed=1)
    p["grid"] = np.zeros_like(p["grid"])
    for a in p["weights"] + p["biases"]:
        a[:] = 0.0
    p["weights"][0][0, :4] = [scale, scale / 16, scale / 256, 1.0]
    p["weights"][1][0, 0] = 1.0
    i = np.arange(17 ** 3)
    v = np.stack([i % 17, i // 17 % 17, i // 289], 1)
    pts = (v / 16.0).astype(np.float32)
    arg = pts.astype(np.float64) @ np.array([scale, scale / 16, scale / 256])
    want = np.cos(arg)
    net, x = S.Network(p, max_fit_points=len(i)), torch.tensor(pts, device="cuda")
    if path == "backward":
        g, w, b = (torch.empty_like(t) for t in (net.grid, net.weights, net.biases))
        S.srn_backward(net.ctx, x, torch.ones((len(i), 1), device="cuda"), g, w, b)
        got = g.cpu().numpy().reshape(-1, 4)[:, 0]  # vertex order is x fastest, as i
    else:
        rho, grad = torch.empty(len(i), device="cuda"), torch.empty((len(i), 3), device="cuda")
        S.srn_density_grad(net.ctx, x, rho, grad)
        got = grad.cpu().numpy()[:, 0] / scale
    rms = lambda e: float(np.sqrt(np.mean(e ** 2)))  # noqa: E731
    assert rms(got - want) <= 1.45 * rms(want.astype(np.float32) - want)


@pytest.mark.parametrize("act,most", [(synth.ACT_SINE, 1.08e-7), (synth.ACT_SNAKEALT, 1.395e-7)])
def test_position_gradient_rounds_each_fourier_row_once(S, act, most):
    """Two-layer networks without latent values: the error of the position
    gradient against 64 bits, relative to its norm, mean of six networks.  One
    thread adding the Fourier rows by FMAs has 1.059e-7 and 1.384e-7, sums of
    four lanes' products 1.116e-7 and 1.410e-7."""
    import torch
    errs = []
    for seed in range(6):
        p = synth.random_params(R=4, F=4, m=12, layers=2, width=32, act=act, seed=seed, bias_std=0.1)
        p["grid"] = np.zeros_like(p["grid"])
        net, pts = S.Network(p), _points(20000, seed)
        rho, grad = torch.empty(20000, device="cuda"), torch.empty((20000, 3), device="cuda")
        S.srn_density_grad(net.ctx, torch.tensor(pts, device="cuda"), rho, grad)
        want = oracle.net_input_grad(oracle.OracleNet(p), pts)[1]
        errs.append(np.linalg.norm(grad.cpu().numpy() - want) / np.linalg.norm(want))
    assert np.mean(errs) <= most


# (width, layers, latent channels, Fourier rows, outputs, time input, NeRF matrix): inputs at both sides of the line
# past which layer 0 runs in blocks (128), blocks full and not, with and without Fourier rows
BLOCKED = [(32, 3, 64, 30, 1, 1, True), (32, 3, 68, 30, 1, 0, True), (32, 2, 200, 0, 4, 0, True), (48, 3, 4, 96, 4, 1, False),
           (64, 2, 64, 93, 1, 0, False), (64, 8, 32, 110, 1, 0, False), (32, 8, 4, 124, 4, 1, False)]


@pytest.mark.parametrize("n", [33, 700])
@pytest.mark.parametrize("width,layers,F,m,D,ti,nerf", BLOCKED)
def test_wide_inputs_match_oracle(S, width, layers, F, m, D, ti, nerf, n):
    """Outputs and density gradient to the FP32 bounds of the oracle's
    first-order analysis, the gradient seeded with output adjoints to 1e-4 of
    max(|g|, 1), and the error grid to twice the largest density bound."""
    import torch
    p = synth.random_params(R=5, F=F, m=m, layers=layers, width=width, out_dim=D, act=synth.ACT_SNAKEALT, seed=n, grid_std=0.5,
                            time_input=ti)
    if not nerf:
        p["fourier"] = np.random.default_rng(5).normal(0, 6, (m, 3)).astype(np.float32)
    net, on, pts, t = S.Network(p), oracle.OracleNet(p), _points(n, n), 0.25
    x = torch.tensor(pts, device="cuda")
    brho, bgrad = oracle.error_bounds(on, pts, oracle.PREC_FP32, t)
    out, rho, grad = (torch.full(s, float("nan"), device="cuda") for s in ((n, D), (n,), (n, 3)))
    S.srn_eval(net.ctx, x, out, time=t)
    S.srn_density_grad(net.ctx, x, rho, grad, time=t)
    rref, gref = oracle.net_input_grad(on, pts, t)
    assert torch.equal(rho, out[:, 0])
    assert (np.abs(rho.cpu().numpy() - rref) / np.asarray(brho).reshape(n, -1)[:, 0]).max() <= 1.0
    assert (np.abs(grad.cpu().numpy() - gref) / bgrad).max() <= 1.0
    dout = np.random.default_rng(n + 9).standard_normal((n, D), dtype=np.float32)
    S.srn_input_backward(net.ctx, x, torch.tensor(dout, device="cuda"), grad, time=t)
    vref = oracle.net_input_vjp(on, pts, dout, t)
    assert (np.abs(grad.cpu().numpy() - vref) / np.maximum(np.abs(vref).max(axis=1, keepdims=True), 1.0)).max() <= 1e-4
    vol, err = np.random.default_rng(1).random((6, 7, 8), dtype=np.float32), torch.full((6 ** 3,), float("nan"), device="cuda")
    S.srn_error_grid(net.ctx, torch.tensor(vol, device="cuda"), 6, 2, 3, err, time=t)
    eref = oracle.error_grid(on, vol, 6, 2, 3, t)
    assert np.abs(err.cpu().numpy() - eref.ravel()).max() <= 2.0 * float(np.max(brho)) + 1e-6


def test_wide_inputs_keep_the_warps_of_an_sm(S):
    """255 inputs against 127 of the same eight layers of 64: a quarter more
    arithmetic, and no more than 1.6 times the time (one warp an SM for the
    rows of all inputs: above 2)."""
    import torch
    times = []
    for m in (46, 110):
        p = synth.random_params(R=5, F=32, m=m, layers=8, width=64, act=synth.ACT_SNAKEALT, seed=m, grid_std=0.5)
        p["fourier"] = np.random.default_rng(5).normal(0, 6, (m, 3)).astype(np.float32)
        net, x, out = S.Network(p), torch.tensor(_points(200000, 1), device="cuda"), torch.empty((200000, 1), device="cuda")
        each = []
        for _ in range(9):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            S.srn_eval(net.ctx, x, out)
            t1.record()
            torch.cuda.synchronize()
            each.append(t0.elapsed_time(t1))
        times.append(sorted(each)[4])
    print(f"127 inputs {times[0]:.3f} ms, 255 inputs {times[1]:.3f} ms")
    assert times[1] <= 1.6 * times[0]


@pytest.mark.parametrize("F,most", [(32, 2.2), (64, 3.6)])
def test_gradients_of_many_channels(S, F, most):
    """300,000 points of a two-layer network of 14 Fourier rows: the gradient
    with F latent channels against 16 of them.  Twice the gathers and a third
    more inputs, or four times and twice: a thread per point takes 1.7 and 2.7
    times as long, four channels a pass through little L1 2.5 and 4.6."""
    import torch
    times = []
    for channels in (16, F):
        p = synth.random_params(R=12, F=channels, m=14, layers=2, width=32, act=synth.ACT_SNAKEALT, seed=1, grid_std=0.5)
        net, x = S.Network(p), torch.tensor(_points(300000, 1), device="cuda")
        rho, grad, each = torch.empty(300000, device="cuda"), torch.empty((300000, 3), device="cuda"), []
        for _ in range(9):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            S.srn_density_grad(net.ctx, x, rho, grad)
            t1.record()
            torch.cuda.synchronize()
            each.append(t0.elapsed_time(t1))
        times.append(sorted(each)[4])
    print(f"16 channels {times[0]:.3f} ms, {F} channels {times[1]:.3f} ms")
    assert times[1] <= most * times[0]
