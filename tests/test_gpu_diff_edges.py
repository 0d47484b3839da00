"""The float splat and its adjoint where their kernels have edges, against the FP64 oracle: image sizes that
cut tiles, strips and blocks, blobs from the smallest to ones listed as large (and a full list's
neighbours), one point, views beyond one group of eight, enough of them to be split over blocks,
more tiles than a block's shared memory counts, and weights that are not finite (they must not leave
their own discs)."""
import numpy as np
import pytest
import torch

from oracle import diff_oracle as D
from paper_0811_2055_gb300 import synth

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-30))


def _cams(nv, W, H):
    a = 2.4 * np.arange(nv)
    return [synth.look_at((0.5 + 1.4 * np.cos(t), 0.5 + 0.3 * np.sin(3 * t), 0.5 + 1.4 * np.sin(t)), (0.5, 0.5, 0.5),
                          width=W, height=H) for t in a]


@pytest.mark.parametrize("n,nv,W,H,big", [(1, 1, 64, 16, 0), (700, 1, 65, 17, 0), (1500, 9, 61, 35, 0), (300, 40, 33, 50, 0),
                                          (1031, 2, 130, 7, 0), (60, 2, 300, 260, 20), (40, 1, 4200, 3100, 1)])
def test_image_and_gradients_match_fp64(n, nv, W, H, big):
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    rng = np.random.default_rng(n + W)
    cams = _cams(nv, W, H)
    xyz = rng.uniform(0.2, 0.8, (n, 3)).astype(np.float32)
    w = rng.uniform(-1.0, 2.0, n).astype(np.float32)
    sig = np.exp(rng.uniform(np.log(0.2), np.log(12.0), n))  # some below sigma_min
    sig[:big] = rng.uniform(20.0, 140.0, big)                # some above sigma_max
    logh = np.log(sig * 1.4 / cams[0]["f_px"]).astype(np.float32)
    g = rng.normal(size=(nv, H, W)).astype(np.float32)
    r = G.Renderer()
    img = G.diff_render(r, *to_dev(xyz, w, logh), cams).cpu().numpy()
    gx, gw, gl = (t.cpu().numpy() for t in G.diff_backward(r, *to_dev(xyz, w, logh), cams, to_dev(g)[0]))
    P, Wt, Lh = xyz.astype(np.float64), w.astype(np.float64), logh.astype(np.float64)
    want = np.stack([D.forward(c, P, Wt, Lh) for c in cams])
    sums = [D.backward(c, P, Wt, Lh, g[v].astype(np.float64)) for v, c in enumerate(cams)]
    wx, ww, wl = (sum(s[k] for s in sums) for k in range(3))
    # fp32 projection and sums: the suite's bounds for the image (1e-4) and the adjoint (1e-3)
    assert _rel(img, want) < 1e-4 and np.abs(img - want).max() <= 1e-4 * np.abs(want).max()
    assert _rel(gx, wx) < 1e-3 and _rel(gw, ww) < 1e-3 and _rel(gl, wl) < 1e-3
    r.close()


def test_weights_that_are_not_finite_stay_in_their_discs():
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    cam = _cams(1, 96, 80)[0]
    rng = np.random.default_rng(3)
    xyz = rng.uniform(0.3, 0.7, (200, 3)).astype(np.float32)
    w = np.ones(200, np.float32)
    logh = np.full(200, np.log(2.0 * 1.4 / cam["f_px"]), np.float32)
    r = G.Renderer()
    good = G.diff_render(r, *to_dev(xyz, w, logh), [cam]).cpu().numpy()[0]
    w[0], w[1] = np.nan, np.inf
    img = G.diff_render(r, *to_dev(xyz, w, logh), [cam]).cpu().numpy()[0]
    bad = ~np.isfinite(img)
    inside = np.zeros_like(bad)
    for i in range(2):  # the two discs, with a margin of 1e-3 px for the fp32 centre
        one = D.forward(cam, xyz[i:i + 1].astype(np.float64), np.ones(1), logh[i:i + 1].astype(np.float64))
        inside |= one > 0
        assert bad[one > 1e-6 * one.max()].all()
    assert 20 < bad.sum() <= inside.sum() + 2
    w[:2] = 0.0
    rest = G.diff_render(r, *to_dev(xyz, w, logh), [cam]).cpu().numpy()[0]
    assert np.array_equal(np.isfinite(rest), np.ones_like(bad)) and np.allclose(img[~bad], rest[~bad], rtol=1e-5,
                                                                               atol=1e-6 * good.max())
    r.close()
