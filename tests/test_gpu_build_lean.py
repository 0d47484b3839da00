"""Builds from the library's pool that do not get the memory of a roomy build start over leanly; those of very many
particles are lean from the first.  The trees are the same."""
import pytest
import torch

from paper_0811_2055_gb300 import synth

pytestmark = pytest.mark.gpu


def _particles(n):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    xyz = torch.rand(n, 3, generator=gen, device="cuda")
    return xyz, torch.ones(n, device="cuda"), torch.full((n,), 5e-4, device="cuda")


def _frame(G, tree):
    cam = synth.look_at((0.5, 0.5, -0.4), (0.5, 0.5, 0.5), width=640, height=360)
    r = G.Renderer()
    _, acc = r.render(tree, cam, G.make_params(lambda_px=60.0), image=None)
    i = tree.info()
    out = acc.clone(), (int(i.n_nodes), int(i.n_points), int(i.depth_max))
    r.close()
    return out


def test_a_build_without_room_starts_over_leanly():
    """60M particles with 5.0 GB free: a roomy build takes 5.6 GB, a lean one 4.0."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    parts = _particles(60_000_000)
    t = G.build_lod(*parts)
    want, info = _frame(G, t)
    t.free()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    G.trim_cache(0)
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - 5_000_000_000, dtype=torch.uint8, device="cuda")
    try:
        t = G.build_lod(*parts)
        free, _ = torch.cuda.mem_get_info()
    finally:
        del hold
        torch.cuda.empty_cache()
    got, again = _frame(G, t)
    assert again == info and torch.equal(got, want)
    assert free < 1_500_000_000  # the memory was short
    t.free()
    G.trim_cache(0)


def test_builds_of_very_many_particles_are_lean():
    """2^28 particles and one: the pool holds 66 bytes a particle, and some, after the build, not 94."""
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    n = (1 << 28) + 1
    parts = _particles(n)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    G.trim_cache(0)
    before, _ = torch.cuda.mem_get_info()
    t = G.build_lod(*parts)
    after, _ = torch.cuda.mem_get_info()
    assert before - after < 80 * n
    i = t.info()
    assert int(i.n_particles) == n and int(i.n_points) > n
    t.free()
    G.trim_cache(0)
