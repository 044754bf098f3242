"""Cell sort and latent-grid gradient at the sizes where they change route:
one-pass, bucket and general radix sorts (512 and 2^18 cells), sparse and
dense cells, every channel count, and points crowded into few cells (several
chunks of one bucket), against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2112_01579_gb300 import synth

pytestmark = pytest.mark.gpu

TOL_GRAD = 2e-5  # of the largest entry: the bound of the other FP32 gradient tests


@pytest.fixture(scope="module")
def S():
    from paper_2112_01579_gb300 import build
    build.build()
    from paper_2112_01579_gb300 import srn
    return srn


@pytest.mark.parametrize("R,F,n,crowd", [(3, 8, 1, False), (9, 4, 1025, False), (9, 32, 40000, False), (10, 16, 1024, False),
                                         (10, 8, 33000, True), (33, 16, 3, False), (33, 16, 40000, False),
                                         (33, 32, 20000, True), (42, 4, 5000, True), (65, 4, 2049, False), (66, 4, 5000, False)])
def test_grid_gradient(S, R, F, n, crowd):
    import torch
    p = synth.random_params(R=R, F=F, m=3, layers=2, width=32, act=synth.ACT_SINE, seed=R, grid_std=0.5)
    net = S.Network(p, max_fit_points=max(n, 2))
    rng = np.random.default_rng(n)
    pts = rng.random((n, 3), dtype=np.float32)
    if crowd:  # nine points of ten inside a box of about one cell, at its corner of the domain and off it
        pts[: 9 * n // 10] = (pts[: 9 * n // 10] * (1.2 / (R - 1)) + (2.9 / (R - 1) if R > 10 else 0.0)).astype(np.float32)
    dout = rng.standard_normal((n, 1), dtype=np.float32)
    g, w, b = (torch.full_like(t, float("nan")) for t in (net.grid, net.weights, net.biases))
    S.srn_backward(net.ctx, torch.tensor(pts, device="cuda"), torch.tensor(dout, device="cuda"), g, w, b)
    rg = np.asarray(oracle.net_backward(oracle.OracleNet(p), pts, dout)[2]).ravel()
    got = g.cpu().numpy()
    assert np.abs(got - rg).max() <= TOL_GRAD * np.abs(rg).max()
    assert not got[rg == 0.0].any()
    again = torch.empty_like(g)
    S.srn_backward(net.ctx, torch.tensor(pts, device="cuda"), torch.tensor(dout, device="cuda"), again, w, b)
    assert torch.equal(g, again)  # fixed orders: the same bits on every run


def _shifted(t):
    """A copy of t that starts 16 bytes behind a 512-byte boundary."""
    import torch
    k = 16 // t.element_size()
    v = torch.empty(t.numel() + k, dtype=t.dtype, device=t.device)[k:]
    v.copy_(t.reshape(-1))
    assert v.data_ptr() % 32 == 16
    return v


@pytest.mark.parametrize("F,m,layers,act,keys", [(8, 12, 2, synth.ACT_SINE, 1), (16, 14, 2, synth.ACT_SNAKEALT, 1),
                                                 (16, 14, 4, synth.ACT_SNAKEALT, 1), (16, 14, 4, synth.ACT_SNAKEALT, 3),
                                                 (32, 6, 3, synth.ACT_SNAKEALT, 1), (4, 6, 3, synth.ACT_SINE, 1)])
def test_grids_off_a_32_byte_boundary(S, F, m, layers, act, keys):
    """Grids are 16-byte aligned by contract; those that are not 32-byte
    aligned take narrower gathers and give the same bits."""
    import torch
    p = synth.random_params(R=6, F=F, m=m, layers=layers, width=32, act=act, seed=F + layers, grid_std=0.5, n_keyframes=keys)
    rng = np.random.default_rng(8)
    pts = torch.tensor(rng.random((400, 3), dtype=np.float32), device="cuda")
    dout = torch.tensor(rng.standard_normal((400, 1), dtype=np.float32), device="cuda")
    vol = torch.tensor(rng.random((9, 8, 7), dtype=np.float32), device="cuda")
    t = 0.5 if keys > 1 else 0.0
    got = []
    for shift in (False, True):
        net = S.Network(p, max_fit_points=400, adam=True)
        grid = _shifted(net.grid) if shift else net.grid
        prm = net._params()
        prm.grid = grid.data_ptr()
        S.srn_set_params(net.ctx, prm)
        out, grad, err, loss = (torch.zeros(n, device="cuda") for n in (400, 1200, 125, 1))
        S.srn_density_grad(net.ctx, pts, out, grad, time=t)
        vjp, dg, dw, db = torch.empty_like(grad), torch.empty_like(net.grid), torch.empty_like(net.weights), torch.empty_like(net.biases)
        S.srn_input_backward(net.ctx, pts, dout, vjp, time=t)
        S.srn_backward(net.ctx, pts, dout, dg, dw, db, time=t)
        S.srn_error_grid(net.ctx, vol, 5, 2, 3, err, time=t)
        S.srn_fit_step(net.ctx, vol, 400, 5, 0, loss, time=t)
        half = S.Network(p, precision=S.SRN_PREC_FP16) if (F, m) in ((8, 12), (16, 14)) else None
        rho = torch.zeros((400, 1), device="cuda")
        if half is not None:
            prm = half._params()
            grid_h = _shifted(half.grid_h) if shift else half.grid_h
            prm.grid_h = grid_h.data_ptr()
            S.srn_set_params(half.ctx, prm)
            S.srn_eval(half.ctx, pts, rho, time=t)
        torch.cuda.synchronize()
        got.append([x.clone() for x in (out, grad, vjp, dg, dw, db, err, loss, grid, net.weights, net.biases, rho)])
    for a, b in zip(*got):
        assert torch.equal(a, b)


def _crowd(kind, n, k, R, seed):
    """n points, k of them in one place below the middle: a `cell`, the cells
    of one leading `digit` of the cell index (three rows of a z layer at R =
    33), or `two` cells a half of the grid apart; the others above the middle."""
    rng = np.random.default_rng(seed)
    pts, h = rng.random((n, 3), dtype=np.float32), 1.0 / (R - 1)
    u = 0.02 + 0.96 * pts[:k].astype(np.float64)
    pts[k:, 2] = 0.5 + 0.5 * pts[k:, 2]
    if kind == "cell":
        pts[:k] = (u + [2, 1, 1]) * h
    elif kind == "two":
        u[::2, 2] += R // 2
        pts[:k] = (u + [1, 2, 0]) * h
    else:
        pts[:k] = np.stack([u[:, 0] * (R - 1), u[:, 1] * 3 + R // 2, u[:, 2] + R // 3], 1) * h
    return rng.permutation(np.clip(pts, 0.0, 1.0), axis=0).astype(np.float32)


@pytest.mark.parametrize("R,F,n,k,kind", [(5, 16, 1900, 1800, "cell"), (10, 8, 20000, 18000, "cell"), (10, 8, 131073, 65536, "cell"),
                                          (10, 4, 131073, 65537, "cell"), (17, 32, 20000, 18000, "two"),
                                          (33, 16, 131072, 131000, "cell"), (33, 16, 300001, 270000, "cell"),
                                          (33, 8, 140000, 131072, "digit"), (33, 4, 300000, 270000, "two"),
                                          (42, 4, 140000, 120000, "digit"), (65, 8, 20000, 18000, "cell"),
                                          (65, 4, 180000, 160000, "two")])
def test_crowded_points(S, R, F, n, k, kind):
    """Cells of more points than a warp takes and leading digits of more keys
    than a block sorts: whole at the limit and cut one past it, segments full
    and not, up to 27 of them, one and two cut digits, eight and ten low bits,
    and what the static scratch holds of it."""
    import torch
    p = synth.random_params(R=R, F=F, m=3, layers=2, width=32, act=synth.ACT_SINE, seed=R, grid_std=0.5)
    net, rng = S.Network(p, max_fit_points=n), np.random.default_rng(n)
    pts, dout = _crowd(kind, n, k, R, n), rng.standard_normal((n, 1), dtype=np.float32)
    x, d = torch.tensor(pts, device="cuda"), torch.tensor(dout, device="cuda")
    rg = np.asarray(oracle.net_backward(oracle.OracleNet(p), pts, dout)[2]).ravel()
    g, w, b = (torch.full_like(t, float("nan")) for t in (net.grid, net.weights, net.biases))
    S.srn_backward(net.ctx, x, d, g, w, b)
    assert np.abs(g.cpu().numpy() - rg).max() <= TOL_GRAD * np.abs(rg).max()
    again = torch.full_like(g, float("nan"))
    S.srn_backward(net.ctx, x, d, again, w, b)
    assert torch.equal(g, again)
    if n * F <= 1200000:
        S.srn_backward_static(net.cfg, net._params(), x, d, again, w, b)
        assert np.abs(again.cpu().numpy() - rg).max() <= TOL_GRAD * np.abs(rg).max()


@pytest.mark.parametrize("kind,F,m,most", [("cell", 16, 14, 20), ("two", 16, 14, 20), ("digit", 8, 12, 3)])
def test_crowded_points_take_their_share_of_the_chip(S, kind, F, m, most):
    """2^18 points of a two-layer network, all in one cell, pair of cells or
    leading digit, against the evenly spread batch.  A cell: within 20 times
    (a warp per vertex over the points of its cells takes 19 times, one warp
    on all points of a cell 196).  A digit's cells: within 3 times (1.7 with a
    sort that does not look at the digits, 4.8 with one block per digit)."""
    import torch
    n = 1 << 18
    p = synth.random_params(R=33, F=F, m=m, layers=2, width=32, act=synth.ACT_SNAKEALT, seed=1, grid_std=0.5)
    net = S.Network(p, max_fit_points=n)
    d = torch.randn((n, 1), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    g, w, b = (torch.empty_like(t) for t in (net.grid, net.weights, net.biases))

    def us(pts):
        x, times = torch.tensor(pts, device="cuda"), []
        for _ in range(12):
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record()
            S.srn_backward(net.ctx, x, d, g, w, b)
            t1.record()
            torch.cuda.synchronize()
            times.append(1e3 * t0.elapsed_time(t1))
        return sorted(times)[len(times) // 2]

    even, crowded = us(np.random.default_rng(1).random((n, 3), dtype=np.float32)), us(_crowd(kind, n, n, 33, 1))
    print(f"{kind}: {even:.0f} us evenly spread, {crowded:.0f} us crowded")
    assert crowded <= most * even


@pytest.mark.parametrize("R,F,points,cells_held", [(17, 16, 1000, True), (65, 16, 5000, True), (83, 16, 5000, False), (17, 4, 140000, True)])
def test_scratch_is_what_the_header_says(S, R, F, points, cells_held):
    """Device memory of a context: per-cell sums of 32 F (R - 1)^3 bytes up to
    256 MB, and at most 32 F + 200 bytes a point, three times the parameters
    and 64 MB of fixed arrays and allocation granularity beside them."""
    import ctypes

    import torch
    p = synth.random_params(R=R, F=F, m=3, layers=2, width=32, act=synth.ACT_SINE, seed=1)
    keep = S.Network(p, max_fit_points=0)  # the parameters, before the count
    cfg = keep.cfg
    cfg.max_fit_points = points
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = S.srn_create(cfg, keep._params())
    held = before - torch.cuda.mem_get_info()[0]
    assert isinstance(ctx, ctypes.c_void_p)
    S.srn_destroy(ctx)
    cells = 32 * F * (R - 1) ** 3
    rest = (32 * F + 200) * points + 3 * 4 * keep.grid.numel() + (64 << 20)
    assert held <= (cells if cells_held else 0) + rest
    assert held >= (cells if cells_held else 0)
