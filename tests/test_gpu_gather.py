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
