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
