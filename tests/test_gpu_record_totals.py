"""Passes with 2^32 (tile, splat) records and more: their number is known in 64 bits, so the pass is split and no
record is placed outside the buffer.  Identical points, so the image is known: their number times one point's."""
import math

import pytest
import torch

from paper_0811_2055_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1 << 20, (1 << 20) + 4097])
@pytest.mark.parametrize("sigma_px", [64.0, 0.25])
def test_all_particle_frames(n, sigma_px):
    """Tiles of one pixel: 64 x 64 of them, all reached by every blob of 64 px (4,096 n records: 2^32, or a little more);
    or boxes of a few pixels, in the small-box stream (a record per pixel: 9 n)."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    cam = synth.look_at((0.5, 0.5, -1.0), (0.5, 0.5, 0.5), width=64, height=64)
    par = G.make_params(tile_w=1, tile_h=1, sigma_min_px=0.25)
    xyz = torch.full((n, 3), 0.5, device="cuda")
    one = torch.ones(n, device="cuda")
    h = one * (sigma_px * 1.5 / cam["f_px"])
    r = G.Renderer()
    _, want = r.render_bruteforce(xyz[:1], one[:1], h[:1], cam, par, image=None)
    want = want.clone()
    assert int(want.max()) > 0 and int(want.max()) < 2 ** 42
    _, acc = r.render_bruteforce(xyz, one, h, cam, par, image=None)
    torch.cuda.synchronize()
    assert r.status() == G.OK and r.stats()["pairs"] == (4096 * n if sigma_px > 1 else 0)
    assert torch.equal(acc, want * n)
    r.close()


def test_float_splats():
    """2^21 points of two views, each reaching the 1,024 tiles of a 1 x 16384 image: 2^32 records.  A pixel is the sum of
    2^21 equal terms, in 32 bits: a unit's at most 1,024 after one another, then 2,048 or fewer units' sums, each rounded to
    2^-24: (1024 + 2048) 2^-24 < 2e-4."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    n = 1 << 21
    cams = [synth.look_at((0.5, 0.5, z), (0.5, 0.5, 0.5), width=1, height=16384) for z in (-1.0, 2.0)]
    par = G.make_params(sigma_max_px=4096.0)
    xyz = torch.full((n, 3), 0.5, device="cuda")
    w = torch.ones(n, device="cuda")
    logh = torch.full((n,), 10.0, device="cuda")  # at the largest sigma
    r = G.Renderer()
    want = G.diff_render(r, xyz[:1], w[:1], logh[:1], cams, par).double() * n
    got = G.diff_render(r, xyz, w, logh, cams, par).double()
    assert float(want.min()) > 0.0
    assert float(((got - want).abs() / want).max()) < 2e-4
    r.close()


@pytest.mark.parametrize("n, nv", [(1 << 21, 40), (3_000_017, 23)])
def test_float_splats_of_several_view_chunks(n, nv):
    """More than 2^26 (view, point) pairs: the views of a call equal the same views alone (up to the sums' order)."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    xyz = 0.2 + 0.6 * torch.rand(n, 3, generator=g, device="cuda")
    w = torch.rand(n, generator=g, device="cuda")
    a = [0.3 * k for k in range(nv)]
    cams = [synth.look_at((0.5 + 1.4 * math.cos(t), 0.5, 0.5 + 1.4 * math.sin(t)), (0.5, 0.5, 0.5), width=40, height=24)
            for t in a]
    logh = torch.full((n,), math.log(0.7 * 1.4 / cams[0]["f_px"]), device="cuda")
    r = G.Renderer()
    got = G.diff_render(r, xyz, w, logh, cams)
    for v in (0, nv // 2, nv - 1):
        one = G.diff_render(r, xyz, w, logh, [cams[v]])[0]
        # positive terms in 32 bits: items of up to 1,024 records, then at most n / 128 items, on either side
        assert float((got[v] - one).abs().max()) <= 2 * (1024 + n / 128) * 2.0 ** -24 * float(one.max())
    r.close()
