"""Gradients where a weight, an upstream value or their products are not finite: the per-pixel terms
decide, as summed one by one (a pixel whose upstream value is zero adds nothing)."""
import numpy as np
import pytest
import torch

from paper_0811_2055_gb300 import synth

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

W, H = 130, 90
SIZES = [1.0, 6.0, 60.0]  # px: discs taken by a group, by a warp, and listed as large


def _terms(cam, xyz, w, logh, g):
    """The adjoint of one point's float splat, pixel by pixel in float32."""
    f = np.float32
    d = xyz.astype(f) - np.asarray(cam["eye"], f)
    xc, yc, zc = (f(np.dot(np.asarray(cam[k], f), d)) for k in ("right", "up", "fwd"))
    F = f(cam["f_px"])
    iz = f(1) / zc
    u, v = f(cam["cx"]) + F * xc * iz, f(cam["cy"]) - F * yc * iz
    raw = F * np.exp(f(logh)) * iz
    s = np.clip(raw, f(0.5), f(128.0))
    y, x = np.mgrid[0:H, 0:W]
    dx, dy = x.astype(f) + f(0.5) - u, y.astype(f) + f(0.5) - v
    r2, s2 = dx * dx + dy * dy, s * s
    norm, e45 = f(0.16951204) / s2, f(np.exp(-4.5))
    e = np.exp(-r2 / (f(2) * s2)) * norm
    k = e - e45 * norm
    on = (r2 < f(9) * s2) & (g != 0)
    gw = g * f(w)
    t = [np.where(on, a, f(0)).sum(dtype=np.float64)
         for a in (g * k, gw * e * dx / s2, gw * e * dy / s2, gw * (e * r2 / (s2 * s) - f(2) * k / s))]
    free = f(0.5) <= raw <= f(128.0)
    return t[0], t[3] * s if free else 0.0, on.any()


def _run(sig, w0, plant):
    """Gradients of 40 points, point 0 (disc of `sig` px around the image's middle) with weight w0; plant(g, u, v) edits
    the upstream image."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    cam = synth.look_at((0.5, 0.5, -1.0), (0.5, 0.5, 0.5), width=W, height=H)
    rng = np.random.default_rng(int(sig * 10))
    xyz = rng.uniform(0.3, 0.7, (40, 3)).astype(np.float32)
    xyz[0] = (0.503, 0.497, 0.5)
    logh = np.full(40, np.log(1.5 * 1.5 / cam["f_px"]), np.float32)
    logh[0] = np.log(sig * 1.5 / cam["f_px"])
    w = rng.uniform(0.5, 1.0, 40).astype(np.float32)
    w[0] = w0
    g = rng.uniform(0.5, 1.5, (1, H, W)).astype(np.float32)
    plant(g[0])
    r = G.Renderer()
    out = [t.cpu().numpy() for t in G.diff_backward(r, *to_dev(xyz, w, logh), [cam], to_dev(g)[0])]
    r.close()
    with np.errstate(all="ignore"):
        want = _terms(cam, xyz[0], w[0], logh[0], g[0])
    return out, want, (xyz, w, logh, g, cam)


@pytest.mark.parametrize("sig", SIZES)
@pytest.mark.parametrize("w0", [np.inf, -np.inf, np.nan, 3e38])
def test_a_zero_upstream_gives_zero(sig, w0):
    (gx, gw, gl), want, _ = _run(sig, w0, lambda g: g.fill(0.0))
    assert want == (0.0, 0.0, False)
    assert not gx.any() and not gw.any() and not gl.any()  # NaN counts as true


@pytest.mark.parametrize("sig", SIZES)
@pytest.mark.parametrize("bad", [np.inf, -np.inf])
def test_an_infinite_upstream_value(sig, bad):
    """At the disc's middle pixel, inside this disc and others: k > 0 there, so dL/dw has the value's sign; r^2 is
    small, so dL/dlog h has the other."""
    def plant(g):
        g[H // 2, W // 2] = bad
    (gx, gw, gl), want, _ = _run(sig, 1.0, plant)
    assert want[0] == bad and want[1] == -bad and want[2]
    assert gw[0] == bad and gl[0] == -bad


@pytest.mark.parametrize("sig", SIZES)
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_what_lies_outside_a_disc_adds_nothing(sig, bad):
    def plant(g):
        g[0, 0] = g[H - 1, W - 1] = bad
    (gx, gw, gl), want, _ = _run(sig, 1.0, plant)
    if sig < 20:
        assert np.isfinite(gx).all() and np.isfinite(gw).all() and np.isfinite(gl).all()
        assert abs(gw[0] - want[0]) < 1e-3 * abs(want[0]) and abs(gl[0] - want[1]) < 1e-3 * abs(want[1])
    else:
        assert not np.isfinite(gw[0])


@pytest.mark.parametrize("sig", SIZES)
def test_large_values_whose_terms_are_finite(sig):
    """Plain sums of these upstream values overflow, the terms scaled by the kernel do not."""
    def plant(g):
        g[:] = 2e38 / max(1.0, 40.0 / sig ** 2)
    (gx, gw, gl), want, _ = _run(sig, 1e-30, plant)
    assert np.isfinite(want[0]) and np.isfinite(want[1])
    # the sum of the kernel over the disc is 1: fp32 sums of at most 128^2 terms of one sign
    assert abs(gw[0] - want[0]) < 1e-3 * abs(want[0])


def test_supports_below_the_smallest_square():
    """sigma^2 underflows: the disc holds no pixel, every gradient is zero."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    cam = synth.look_at((0.5, 0.5, -1.0), (0.5, 0.5, 0.5), width=97, height=81)  # the middle is a pixel's centre
    xyz = np.full((3, 3), 0.5, np.float32)
    w, logh = np.ones(3, np.float32), np.full(3, -100.0, np.float32)
    g = np.ones((1, 81, 97), np.float32)
    r = G.Renderer()
    par = G.make_params(sigma_min_px=1e-25)
    for t in G.diff_backward(r, *to_dev(xyz, w, logh), [cam], to_dev(g)[0], par):
        assert not t.cpu().numpy().any()
    assert not G.diff_render(r, *to_dev(xyz, w, logh), [cam], par).cpu().numpy().any()
    r.close()


@pytest.mark.parametrize("w0", [np.inf, 1.0])
def test_more_large_discs_than_the_list_takes(w0):
    """70,000 discs of 8,192 pixels and more (65,536 are listed): with upstream values one call equals two calls of half
    the points; with infinite weights and no upstream values all gradients are zero."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    n = 70_000
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    cam = synth.look_at((0.5, 0.5, -1.0), (0.5, 0.5, 0.5), width=130, height=90)
    xyz = 0.45 + 0.1 * torch.rand(n, 3, generator=gen, device="cuda")
    w = torch.full((n,), float(w0), device="cuda")
    logh = torch.full((n,), float(np.log(70.0 * 1.5 / cam["f_px"])), device="cuda")
    g = torch.randn(1, 90, 130, generator=gen, device="cuda")
    if not np.isfinite(w0):
        g.zero_()
    r = G.Renderer()
    all_ = G.diff_backward(r, xyz, w, logh, [cam], g)
    if not np.isfinite(w0):
        assert not any(bool(t.any()) or bool(t.isnan().any()) for t in all_)
    else:
        m = n // 2
        halves = [G.diff_backward(r, xyz[a:b].contiguous(), w[a:b].contiguous(), logh[a:b].contiguous(), [cam], g)
                  for a, b in ((0, m), (m, n))]
        for t, h in zip(all_, (torch.cat(p) for p in zip(*halves))):
            # sums of 11,700 signed terms in 32 bits, grouped differently
            assert float((t - h).abs().max()) <= 2 * 11700 * 2.0 ** -24 * float(h.abs().max())
    r.close()


@pytest.mark.parametrize("n, nv", [(160_001, 9), (160_001, 17), (40_000, 8)])
@pytest.mark.parametrize("bad", [False, True])
def test_several_views_of_a_point_in_one_block(n, nv, bad):
    """Many points, so that a group of lanes sums its point over eight views and more: the gradients are the sums of
    one-view calls.  bad: an infinite weight without upstream values in some of the views."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n + nv)
    xyz = 0.2 + 0.6 * torch.rand(n, 3, generator=gen, device="cuda")
    w = torch.rand(n, generator=gen, device="cuda")
    a = 2.4 * np.arange(nv)
    cams = [synth.look_at((0.5 + 1.4 * np.cos(t), 0.5 + 0.3 * np.sin(3 * t), 0.5 + 1.4 * np.sin(t)), (0.5, 0.5, 0.5),
                          width=40, height=28) for t in a]
    sig = torch.exp(torch.empty(n, device="cuda").uniform_(-0.7, 1.5, generator=gen))
    logh = torch.log(sig * (1.4 / cams[0]["f_px"]))
    g = torch.randn(nv, 28, 40, generator=gen, device="cuda")
    if bad:
        g[::2] = 0.0
        w[::97] = float("inf")
    r = G.Renderer()
    got = G.diff_backward(r, xyz, w, logh, cams, g)
    ones = [G.diff_backward(r, xyz, w, logh, [cams[v]], g[v:v + 1]) for v in range(nv)]
    for k in range(3):
        parts = torch.stack([o[k] for o in ones]).double()
        want, size = parts.sum(0), parts.abs().sum(0)
        ok = torch.isfinite(want)
        assert torch.equal(ok, torch.isfinite(got[k]))
        # the same terms of a view, then nv of them, in 32 bits in another order
        assert bool(((got[k].double() - want).abs()[ok] <= (2 * nv * 2.0 ** -24 * size + 1e-30)[ok]).all())
    r.close()


@pytest.mark.parametrize("w0", [3e38, -3e38, np.inf])
def test_the_image_of_a_weight_whose_peak_overflows(w0):
    """sigma 0.25 px: the norm is 2.7, so the peak of a weight of 3e38 overflows, but not its flank: the kernel value
    scales the weight first."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    cam = synth.look_at((0.5, 0.5, -1.0), (0.5, 0.5, 0.5), width=64, height=48)
    f = np.float32
    xyz = np.array([[0.5, 0.5, 0.5], [0.6, 0.55, 0.5]], np.float32)
    w, sig = np.array([w0, 1.0], np.float32), f(0.25)
    logh = np.full(2, np.log(0.1 * 1.5 / cam["f_px"]), np.float32)
    r = G.Renderer()
    par = G.make_params(sigma_min_px=0.25)
    img = G.diff_render(r, *to_dev(xyz, w, logh), [cam], par).cpu().numpy()[0]
    unit = G.diff_render(r, *to_dev(xyz, np.array([1.0, 0.0], np.float32), logh), [cam], par).cpu().numpy()[0]
    rest = G.diff_render(r, *to_dev(xyz, np.array([0.0, 1.0], np.float32), logh), [cam], par).cpu().numpy()[0]
    on = unit > 0
    norm = f(0.16951204) / (sig * sig)
    with np.errstate(over="ignore"):
        want = (f(w0) * (unit[on] / norm)) * norm
    assert on.sum() >= 4
    if np.isfinite(w0):
        assert np.isfinite(want).all()  # the centre lies between four pixels
        assert np.allclose(img[on], want, rtol=1e-4)
    else:
        assert (img[on] == np.inf).all()
    assert np.array_equal(img[~on], rest[~on])
    r.close()
