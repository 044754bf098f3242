"""One context used from two streams, and one network from two host threads:
calls that share nothing give the bits of serial calls, and no call leaves
anything behind that a later one trips over."""
import threading

import numpy as np
import pytest

from paper_2112_01579_gb300 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    from paper_2112_01579_gb300 import build
    build.build()
    from paper_2112_01579_gb300 import srn
    return srn


def _frame(S, net, w=200, h=150):
    import torch
    img = torch.full((1, 1, h, w, 4), float("nan"), device="cuda")
    ns = torch.zeros(1, dtype=torch.int64, device="cuda")
    S.srn_render(net.ctx, synth.orbit_cameras(1), synth.tf_preset(8), S.render_desc(w, h, 1 / 128, 0.99), img, samples=ns)
    torch.cuda.synchronize()
    return img, int(ns.item())


@pytest.mark.parametrize("overlap", ["points", "points and frames", "frames"])
def test_overlapping_calls_of_one_fp16_context(S, overlap):
    """Point calls of different sizes on two streams, beside frames or alone,
    give the bits of serial calls; frames that overlap each other share a work
    counter and may be spoilt, but whatever overlapped, every later frame has
    all its pixels and its samples counted once."""
    import torch
    p = synth.to_half_exact(H.cfg2_params(seed=5, R=8))
    net, fresh = S.Network(p, precision=S.SRN_PREC_FP16), S.Network(p, precision=S.SRN_PREC_FP16)
    want, samples = _frame(S, fresh)
    assert torch.isfinite(want).all() and samples > 0
    rng = np.random.default_rng(1)
    sizes = [160, 1000, 33, 100000, 700]
    pts = [torch.tensor(rng.random((n, 3), dtype=np.float32), device="cuda") for n in sizes]
    ref = [torch.empty((n, 1), device="cuda") for n in sizes]
    for x, r in zip(pts, ref):
        S.srn_eval(fresh.ctx, x, r)
    out = [[torch.full_like(r, float("nan")) for r in ref] for _ in range(2)]
    img = [torch.empty((1, 1, 150, 200, 4), device="cuda") for _ in range(2)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    cams, tf, desc = synth.orbit_cameras(1), synth.tf_preset(8), S.render_desc(200, 150, 1 / 128, 0.99)
    small = S.render_desc(40, 30, 1 / 128, 0.99)
    torch.cuda.synchronize()
    for rep in range(100):
        for k, st in enumerate(streams):
            if overlap == "frames" or (overlap == "points and frames" and k == 0):
                S.srn_render(net.ctx, cams, tf, desc if (rep + k) % 2 else small, img[k], stream=st)
            if overlap != "frames":
                for i in range(len(sizes)):
                    j = (i + rep + 2 * k) % len(sizes)
                    S.srn_eval(net.ctx, pts[j], out[k][j], stream=st)
        if rep % 10 == 9:
            torch.cuda.synchronize()
            for _ in range(2):
                got, ns = _frame(S, net)
                assert torch.equal(got, want) and ns == samples, (rep, ns, samples)
    if overlap != "frames":
        for o in out:
            for a, b in zip(o, ref):
                assert torch.equal(a, b)


def test_two_threads_one_network(S):
    """Large and small FP32 batches of one network from two host threads: the
    CTA, and with it the shared memory a launch asks for, follows the batch."""
    import torch
    net = S.Network(H.cfg2_params(seed=6, R=8))
    rng = np.random.default_rng(2)
    vol = torch.tensor(rng.random((9, 8, 7), dtype=np.float32), device="cuda")
    sizes, errors = [60000, 50], []
    pts = [torch.tensor(rng.random((n, 3), dtype=np.float32), device="cuda") for n in sizes]
    out = [[torch.empty((n, 1), device="cuda"), torch.empty((n, 3), device="cuda")] for n in sizes]
    err = [torch.empty(r ** 3, device="cuda") for r in (40, 4)]

    def calls(k, reps, stream):
        try:
            for _ in range(reps):
                S.srn_eval(net.ctx, pts[k], out[k][0], stream=stream)
                S.srn_density_grad(net.ctx, pts[k], out[k][0], out[k][1], stream=stream)
                S.srn_error_grid(net.ctx, vol, 40 if k == 0 else 4, 1, 3, err[k], stream=stream)
        except S.SrnError as e:
            errors.append(str(e))

    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for k in range(2):
        calls(k, 1, streams[k])
    torch.cuda.synchronize()
    want = [x.clone() for x in (*out[0], *out[1], *err)]
    threads = [threading.Thread(target=calls, args=(k, 3000, streams[k])) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[:2]
    for a, b in zip(want, (*out[0], *out[1], *err)):
        assert torch.equal(a, b)
