"""Batches binned in parts (all views' tiles in shared memory, one to four blocks per SM) and through the global
tile counters (more tiles), a captured small batch in scratch reserved for a larger one, and the tone map's passes
at their edges: pixel counts around a block's, accumulators at the ends of the range and of 64 bits."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_0811_2055_gb300 import synth

from gpu_helpers import to_dev, u8_close

pytestmark = pytest.mark.gpu


def _cams(n, W, H):
    eyes = np.random.default_rng(n).uniform(-0.2, 1.2, (n, 3))
    return [synth.look_at(tuple(e), (0.5, 0.5, 0.5), width=W, height=H, z_near=1e-3) for e in eyes]


def _views(tree, cams):
    return [(tree, c, torch.full((c["height"], c["width"]), 3, dtype=torch.uint8, device="cuda"),
             torch.full((c["height"], c["width"]), 77, dtype=torch.int64, device="cuda")) for c in cams]


# tiles in all: 16, 7.5k, 15.4k, 30k (four to one blocks per SM) and 80k (global counters)
@pytest.mark.parametrize("n, W, H, tw, th", [(2, 96, 50, 64, 16), (3, 800, 800, 16, 16), (6, 820, 800, 16, 16),
                                             (3, 800, 800, 8, 8), (8, 800, 800, 8, 8)])
@pytest.mark.parametrize("block16", [False, True])
@pytest.mark.parametrize("kernel", [0, 1])
def test_batches_equal_the_oracle(n, W, H, tw, th, block16, kernel):
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    p = synth.clustered(30011, 48, 0.1, 0.25, seed=n)
    ot = O.build_tree(p.xyz, p.mass, p.h, seed=1, n_max=700)
    t = G.build_lod(*to_dev(p.xyz, p.mass, p.h), n_max=700, seed=1)
    fmt = {}
    if block16:
        t.quantize()
        fmt["point_format"] = G.POINTS_BLOCK16
        ot = O.block_quantize(ot)[2]
    views = _views(t, _cams(n, W, H))
    par = G.make_params(lambda_px=6.0, kernel=kernel, tile_w=tw, tile_h=th, **fmt)
    r = G.Renderer()
    r.reserve_batch(views, par, record_capacity=1 << 28)
    r.render_batch(views, par)
    torch.cuda.synchronize()
    assert r.status() == G.OK
    orp = O.rparams(lambda_px=6.0, kernel=kernel)
    splats = 0
    for _, cam, img, acc in views:
        want, st, nd, _ = O.render_lod(ot, cam, orp)
        splats += nd
        assert st == 0 and np.array_equal(G.u64(acc), want)
        assert u8_close(img.cpu().numpy(), O.tonemap(want, orp)) <= 1
    assert r.stats()["splats"] == splats
    t.free()
    r.close()


def test_small_batch_in_scratch_of_a_large_one():
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    p = synth.tiny(20000, seed=3)
    t = G.build_lod(*to_dev(p.xyz, p.mass, p.h), n_max=400, seed=2)
    par = G.make_params(lambda_px=6.0, tile_w=8, tile_h=8)
    large, small = _views(t, _cams(8, 800, 800)), _views(t, _cams(5, 420, 410))
    r = G.Renderer()
    r.reserve_batch(large, par, record_capacity=1 << 22)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        r.render_batch(small, par)
    s.synchronize()
    want = [(img.clone(), acc.clone()) for _, _, img, acc in small]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        r.render_batch(small, par)
    for _, _, img, acc in small:
        img.zero_()
        acc.zero_()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert r.status() == G.OK
    alone = G.Renderer()
    for (_, cam, img, acc), (wi, wa) in zip(small, want):
        ia, aa = alone.render(t, cam, par)
        assert torch.equal(acc, wa) and torch.equal(img, wi) and torch.equal(acc, aa) and torch.equal(img, ia)
    alone.close()
    r.close()
    t.free()


@pytest.mark.parametrize("n", [1, 255, 2047, 2048, 2049, 7 * 14287])
@pytest.mark.parametrize("lo, hi", [(0.5, 2.0 ** 20), (3.0, 5.0), (2.0 ** 53 + 2, 2.0 ** 60), (2.0 ** 53 + 4, 2.0 ** 54),
                                    (2.0 ** 63 + 2 ** 11, 2.0 ** 64), (2.0 ** 64, 2.0 ** 70), (None, None)])
def test_tone_map_edges(n, lo, hi):
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    rng = np.random.default_rng(n)
    acc = np.exp2(rng.uniform(0.0, 63.9, n)).astype(np.uint64)
    near = [0, 1, 2 ** 64 - 1]
    for v in (lo, hi):
        if v is not None:
            near += [min(max(int(v) + k, 0), 2 ** 64 - 1) for k in range(-3, 4)]
    near = np.array(near, np.uint64)[:n]
    acc[rng.permutation(n)[:len(near)]] = near
    kw = dict(tone_auto=0) if lo is not None else {}
    if lo is not None:
        kw.update(tone_lo=lo / 2.0 ** 32, tone_hi=hi / 2.0 ** 32)
    r = G.Renderer()
    d = torch.from_numpy(acc.view(np.int64).reshape(7 if n > 16384 else 1, -1)).cuda()
    img = r.tonemap(d, G.make_params(**{**kw, "tone_auto": lo is None}))
    assert u8_close(img.cpu().numpy(), O.tonemap(acc.reshape(7 if n > 16384 else 1, -1), O.rparams(**kw))) <= 1
    r.close()


@pytest.mark.parametrize("n", [40, 4000, 60_000])
@pytest.mark.parametrize("size", [(40, 24), (130, 67), (511, 300)])
def test_small_frames_in_small_items(n, size):
    """Records few and many against the work items wanted (below, between and above the bounds of an item's
    size), in one tile and in many, alone and in a batch, against the oracle bit for bit."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    p = synth.tiny(n, seed=n)
    h = p.h * 6.0
    ot = O.build_tree(p.xyz, p.mass, h, seed=1, n_max=900)
    t = G.build_lod(*to_dev(p.xyz, p.mass, h), n_max=900, seed=1)
    views = _views(t, _cams(3, *size))
    par = G.make_params(lambda_px=5.0)
    r = G.Renderer()
    r.reserve_batch(views, par, record_capacity=1 << 24)
    r.render_batch(views, par)
    torch.cuda.synchronize()
    assert r.status() == G.OK
    for _, cam, img, acc in views:
        want, st, nd, _ = O.render_lod(ot, cam, O.rparams(lambda_px=5.0))
        assert st == 0 and np.array_equal(G.u64(acc), want)
        img1, acc1 = r.render(t, cam, par)
        assert torch.equal(acc1, acc) and torch.equal(img1, img)
    t.free()
    r.close()
