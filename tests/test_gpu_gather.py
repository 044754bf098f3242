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
