"""What gblod_renderer_reserve_batch promises: a batch that was not reserved for is refused before anything is
launched, whatever other calls have grown the renderer's buffers to."""
import pytest
import torch

from paper_0811_2055_gb300 import synth

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


def _views(tree, n, W, H):
    out = []
    for k in range(n):
        cam = synth.look_at((0.5, 0.5, -1.0 - 0.1 * k), (0.5, 0.5, 0.5), width=W, height=H)
        out.append((tree, cam, torch.zeros((H, W), dtype=torch.uint8, device="cuda"),
                    torch.zeros((H, W), dtype=torch.int64, device="cuda")))
    return out


def test_larger_batch_after_a_large_frame_is_refused():
    """Eight 1080p views reserved, one 4K frame of 40M particles drawn (its runs of records are counted in groups),
    then eight 4K views: 64,800 tiles go through the global counters, in scratch of 16,320 tiles."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    p = synth.tiny(20000, seed=3)
    t = G.build_lod(*to_dev(p.xyz, p.mass, p.h), n_max=400, seed=2)
    small, large = _views(t, 8, 1920, 1080), _views(t, 8, 3840, 2160)
    par = G.make_params()
    r = G.Renderer()
    r.reserve_batch(small, par, record_capacity=1 << 29)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    n = 40_000_000
    xyz = torch.rand(n, 3, generator=g, device="cuda")
    one = torch.ones(n, device="cuda")
    r.render_bruteforce(xyz, one, 1e-4 * one, large[0][1], par)
    torch.cuda.synchronize()
    launched = G.launch_count()
    with pytest.raises(G.GblodError) as e:
        r.render_batch(large, par)
    assert e.value.code == G.ERR_INVALID_ARG and G.launch_count() == launched
    r.render_batch(small, par)  # what was reserved still runs
    torch.cuda.synchronize()
    assert r.status() == G.OK
    alone = G.Renderer()
    for _, cam, img, acc in small:
        ia, aa = alone.render(t, cam, par)
        assert torch.equal(acc, aa) and torch.equal(img, ia)
    alone.close()
    r.close()
    t.free()


def test_a_captured_batch_survives_other_calls_on_the_renderer():
    """Calls that grow the renderer's own buffers (runs of records in groups, more tiles, deeper trees, fits) between the
    capture of a batch and its replay; none needs more records than were reserved."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    p = synth.tiny(20000, seed=3)
    t = G.build_lod(*to_dev(p.xyz, p.mass, p.h), n_max=400, seed=2)
    deep = G.build_lod(*to_dev(p.xyz, p.mass, p.h), n_max=1, seed=2)
    views = _views(t, 2, 1920, 1080)
    par = G.make_params(lambda_px=6.0)
    r = G.Renderer()
    r.reserve_batch(views, par, record_capacity=1 << 28)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        r.render_batch(views, par)
    s.synchronize()
    want = [(img.clone(), acc.clone()) for _, _, img, acc in views]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        r.render_batch(views, par)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    n = 12_000_000
    xyz = torch.rand(n, 3, generator=gen, device="cuda")
    one = torch.ones(n, device="cuda")
    r.render_bruteforce(xyz, one, 2e-3 * one, views[0][1], par)
    r.render_bruteforce(xyz, one, 1e-4 * one, synth.look_at((0.5, 0.5, -1.0), (0.5, 0.5, 0.5), width=7680, height=4320))
    r.render(deep, views[0][1], G.make_params(lambda_px=0.0))
    G.diff_render(r, xyz[:1000], one[:1000], one[:1000] - 6.0, [views[0][1]])
    torch.cuda.synchronize()
    for _, _, img, acc in views:
        img.zero_()
        acc.zero_()
    torch.cuda.empty_cache()
    graph.replay()
    torch.cuda.synchronize()
    assert r.status() == G.OK
    for (_, _, img, acc), (wi, wa) in zip(views, want):
        assert torch.equal(acc, wa) and torch.equal(img, wi)
    r.close()
    t.free()
    deep.free()


def test_a_batch_whose_records_fit_its_reservation_is_drawn():
    """As many records as make the most work items for their number: a quotient just above an item size (32 tiles,
    all reached by each of 2 want + 66 particles: 64 < records / want < 65), reserved with little to spare."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    n = 2 * 16 * torch.cuda.get_device_properties(0).multi_processor_count + 66
    p = synth.tiny(n, seed=5)
    xyz = (0.5 + 0.01 * (p.xyz - 0.5)).astype("float32")
    t = G.build_lod(*to_dev(xyz, p.mass, 0.0 * p.h + 0.4), n_max=8000, seed=1)
    views = _views(t, 1, 256, 128)
    r = G.Renderer()
    r.reserve_batch(views, record_capacity=1 << 22)
    r.render_batch(views)
    torch.cuda.synchronize()
    assert r.status() == G.OK and r.stats()["pairs"] == 32 * n
    alone = G.Renderer()
    ia, aa = alone.render(t, views[0][1])
    assert torch.equal(views[0][3], aa) and torch.equal(views[0][2], ia)
    alone.close()
    r.close()
    t.free()
