"""Dense DVR and the transfer function at values and views outside the usual
range: infinite and very large voxels, an eye far from the box, negative and
infinite control values."""
import math

import numpy as np
import pytest

import oracle
from paper_2112_01579_gb300 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2112_01579_gb300 import build
    build.build()
    from paper_2112_01579_gb300 import srn
    return srn


def _tf(pos, rgba, scale):
    return dict(pos=np.asarray(pos, np.float32), rgba=np.asarray(rgba, np.float32), opacity_scale=scale)


def _dense(S, vol, cams, tf, w=60, h=44, step=1 / 64, et=0.99, shading=0):
    import torch
    out = torch.full((len(cams), h, w, 4), float("nan"), device="cuda")
    S.srn_dvr_dense(torch.as_tensor(vol, dtype=torch.float32, device="cuda").contiguous(), cams, tf,
                    S.render_desc(w, h, step, et, shading), out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


# one colour above 0.9: a density that interpolation rounds to just below 1 looks like 1
CAPPED = _tf([0.0, 0.5, 0.9, 1.0], [[0, 0, 0, 0], [0.2, 0.7, 0.4, 0.01], [0.9, 0.5, 0.1, 0.05], [0.9, 0.5, 0.1, 0.05]], 20.0)


def test_infinite_voxels_are_opaque(S):
    """+Inf between +Inf is +Inf, the density 1 after the clamp."""
    cams = synth.orbit_cameras(3)
    inf, one = (np.full((9, 10, 11), v, np.float32) for v in (np.inf, 1.0))
    want = _dense(S, one, cams, CAPPED)
    assert want[..., 3].max() > 0.3
    assert np.array_equal(_dense(S, inf, cams, CAPPED), want)


def test_infinite_slab_beside_finite_voxels(S):
    """A slab of +Inf looks like one of 1e30: every weight that is not zero
    takes either of them past 1."""
    cams = synth.orbit_cameras(3)
    vol = synth.blobs_volume(24, 6, seed=3).numpy().copy()
    big, inf = vol.copy(), vol.copy()
    big[8:14], inf[8:14] = 1e30, np.inf
    want = _dense(S, big, cams, CAPPED)
    assert not np.array_equal(want, _dense(S, vol, cams, CAPPED))
    assert np.array_equal(_dense(S, inf, cams, CAPPED), want)


@pytest.mark.parametrize("shading", [0, 2])
@pytest.mark.parametrize("distance", [3.0, 1e4, 1e5])
def test_far_eye_does_not_extrapolate(S, shading, distance):
    """Interpolation stays between the voxels' values whatever the rounding of
    the sample position: nothing outside [0.4, 0.6] is seen.  The outer layer
    differs from the next one, so a position past it would show."""
    rng = np.random.default_rng(4)
    vol = np.where(rng.random((40, 48, 64)) < 0.5, 0.4, 0.6).astype(np.float32)
    vol[0], vol[-1], vol[:, 0], vol[:, -1], vol[:, :, 0], vol[:, :, -1] = (0.6,) * 6
    vol[1], vol[-2], vol[:, 1], vol[:, -2], vol[:, :, 1], vol[:, :, -2] = (0.4,) * 6
    vol[0], vol[-1], vol[:, 0], vol[:, -1], vol[:, :, 0], vol[:, :, -1] = (0.6,) * 6
    marker = _tf([0.0, 0.38, 0.39, 0.61, 0.62, 1.0], [[1, 1, 1, 1]] * 2 + [[0, 0, 0, 0]] * 2 + [[1, 1, 1, 1]] * 2, 500.0)
    d = np.array([0.5, 0.4, 0.77]) / np.linalg.norm([0.5, 0.4, 0.77])
    cams = [dict(eye=list(distance * d), target=[0.0, 0.0, 0.0], up=[0.0, 1.0, 0.0], fovy=2 * math.atan(0.8 / distance))]
    got = _dense(S, vol, cams, marker, 120, 90, 1 / 256, 2.0, shading)
    assert not got.any(), float(np.abs(got).max())
    # the view does hit the volume
    seen = _dense(S, vol, cams, _tf([0.0, 1.0], [[1, 1, 1, 1]] * 2, 20.0), 120, 90, 1 / 256, 2.0, shading)
    assert seen[..., 3].max() > 0.9


@pytest.mark.parametrize("alpha,step", [(-0.4, 0.5), (-0.01, 0.05), (0.4, 0.5)])
def test_negative_alpha_follows_the_exponential(S, alpha, step):
    """1 - exp(-x) for either sign of x.  Constant volume, so the density is
    0.5 to rounding and only the opacity counts: |x| <= 4 a sample to 2^-21
    (product and exponential), at most 40 samples, each factor of the
    transmittance off by 2^-21 (1 + |x|): 5e-5 of the largest value."""
    tf = _tf([0.0, 1.0], [[0.8, 0.5, 0.3, alpha]] * 2, 20.0)
    cams, vol = synth.orbit_cameras(2), np.full((8, 8, 8), 0.5, np.float32)
    got = _dense(S, vol, cams, tf, 40, 30, step, 2.0)
    ref, _, _ = oracle.dvr_dense(vol, cams, H.oracle_tf(tf), 40, 30, step, 2.0)
    assert np.abs(got - ref).max() <= 5e-5 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("path", ["dense", "fp16"])
@pytest.mark.parametrize("where", ["last", "flat", "second"])
def test_infinite_alpha_is_opaque(S, path, where):
    """A control point of infinite alpha stops the ray at its colour; a point
    before it keeps its own."""
    import torch
    alphas = dict(last=[0.0, 0.1, 0.2, np.inf], flat=[0.0, 0.1, np.inf, np.inf], second=[0.0, np.inf, np.inf, np.inf])[where]
    colour = [[0.1, 0.2, 0.3], [0.5, 0.4, 0.3], [0.6, 0.2, 0.9], [0.3, 0.8, 0.7]]
    tfs = [_tf([0.2, 0.4, 0.6, 0.8], [c + [min(a, top)] for c, a in zip(colour, alphas)], 20.0) for top in (np.inf, 1e30)]
    cams = synth.orbit_cameras(2)
    if path == "dense":
        vol = synth.blobs_volume(24, 6, seed=5).numpy()
        got, want = (_dense(S, vol, cams, tf) for tf in tfs)
    else:
        net = S.Network(synth.to_half_exact(H.cfg2_params(seed=8, R=8)), precision=S.SRN_PREC_FP16)
        imgs = []
        for tf in tfs:
            out = torch.full((1, 2, 44, 60, 4), float("nan"), device="cuda")
            S.srn_render(net.ctx, cams, tf, S.render_desc(60, 44, 1 / 64, 0.99), out)
            torch.cuda.synchronize()
            imgs.append(out.cpu().numpy())
        got, want = imgs
    assert want[..., 3].max() == 1.0
    assert np.array_equal(got, want)
