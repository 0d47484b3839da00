"""Passes with 2^32 (tile, splat) records and more: their number is known in 64 bits, so the pass is split and no
record is placed outside the buffer.  Identical points, so the image is known: their number times one point's."""
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
