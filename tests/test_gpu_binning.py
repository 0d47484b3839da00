"""Frames binned in parts (shared-memory histograms) and through the global tile counters, against the oracle
bit for bit: tile counts below and above the shared-memory limit of each point source, fewer points
than one chunk, chunks that end in the middle of a node, record-budget pieces, an octree's fp32 points
and its 16-bit codes, and the caller's unordered arrays."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_0811_2055_gb300 import synth

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 255, 257, 30011])
@pytest.mark.parametrize("W,H,tw,th", [(96, 50, 64, 16), (1800, 1000, 32, 32), (1800, 1000, 8, 8), (1500, 1200, 8, 4)])
@pytest.mark.parametrize("budget", [0, 3000])
def test_binning_equals_the_oracle(n, W, H, tw, th, budget):
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    p = synth.tiny(n, seed=n)
    d = to_dev(p.xyz, p.mass, p.h)
    cam = synth.look_at((0.4, 0.6, -0.7), (0.5, 0.5, 0.5), width=W, height=H)
    ot = O.build_tree(p.xyz, p.mass, p.h, seed=1, n_max=700)
    t = G.build_lod(*d, n_max=700, seed=1)
    r = G.Renderer()
    kw = dict(lambda_px=9.0, tile_w=tw, tile_h=th, record_budget=budget)
    want, st, nd, _ = O.render_lod(ot, cam, O.rparams(lambda_px=9.0))
    _, acc = r.render(t, cam, G.make_params(**kw))
    assert st == 0 and r.status() == G.OK and np.array_equal(G.u64(acc), want)
    assert r.stats()["splats"] == nd
    want, st, nd = O.splat_particles(p.xyz, p.mass, p.h, cam, O.rparams())
    _, acc = r.render_bruteforce(*d, cam, G.make_params(**kw))
    assert st == 0 and r.status() == G.OK and np.array_equal(G.u64(acc), want)
    t.quantize()
    _, _, decoded = O.block_quantize(ot)
    want, st, nd, _ = O.render_lod(decoded, cam, O.rparams(lambda_px=9.0))
    _, acc = r.render(t, cam, G.make_params(point_format=G.POINTS_BLOCK16, **kw))
    assert st == 0 and r.status() == G.OK and np.array_equal(G.u64(acc), want)
    t.free()
    r.close()


@pytest.mark.parametrize("n", [11_200_000, 17_000_001])
def test_records_in_several_regions(n):
    """Enough unordered points for two and three groups of blocks: the same image and counts as through the global
    tile counters."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    g = torch.Generator(device="cuda").manual_seed(n)
    xyz = torch.rand((n, 3), device="cuda", generator=g)
    mass = torch.rand(n, device="cuda", generator=g) + 0.5
    h = torch.rand(n, device="cuda", generator=g) * 0.004 + 1e-4
    cam = synth.look_at((0.4, 0.6, -0.7), (0.5, 0.5, 0.5), width=1500, height=1200)
    r = G.Renderer()
    _, a = r.render_bruteforce(xyz, mass, h, cam, G.make_params(count_updates=True))
    sa = r.stats()
    _, b = r.render_bruteforce(xyz, mass, h, cam, G.make_params(tile_w=8, tile_h=4, count_updates=True))
    sb = r.stats()
    assert r.status() == G.OK and torch.equal(a, b)
    for k in ("points", "splats", "amplitude_lo", "amplitude_hi", "pixel_updates"):
        assert sa[k] == sb[k], k
    r.close()


@pytest.mark.parametrize("side", [0.4, 1.1, 1.9, 2.6, 3.3])
@pytest.mark.parametrize("n", [1, 31, 33, 4095, 4097, 70001])
def test_small_boxes_by_size_equal_the_oracle(side, n):
    """Small boxes of each size alone and together (queues of 4, 6 and 8 pixels that fill, overflow by one and end in
    the middle), all on one pixel and spread out, light and heavy."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    rng = np.random.default_rng(n)
    xyz = rng.uniform(0.0, 1.0, (n, 3)).astype(np.float32)
    xyz[n // 2:] = xyz[0]
    mass = np.exp2(rng.uniform(-12.0, 4.0, n)).astype(np.float32)
    cam = synth.look_at((0.5, 0.5, -1.5), (0.5, 0.5, 0.5), width=130, height=67)
    h = (side / 3.0 * 2.0 / cam["f_px"] * rng.uniform(0.5, 1.0, n)).astype(np.float32)
    r = G.Renderer()
    want, st, nd = O.splat_particles(xyz, mass, h, cam, O.rparams(sigma_min_px=0.25))
    _, acc = r.render_bruteforce(*to_dev(xyz, mass, h), cam, G.make_params(sigma_min_px=0.25))
    assert st == 0 and r.status() == G.OK and np.array_equal(G.u64(acc), want)
    assert r.stats()["splats"] == nd
    r.close()
