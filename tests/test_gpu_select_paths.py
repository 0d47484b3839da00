"""Node selection in one block (at most 256 nodes), flat (at most 2^19) and level by level, alone, in parts
and in batches, against the oracle bit for bit, with frusta that hold all, some and none of the tree."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_0811_2055_gb300 import synth

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu

CAMS = [((0.5, 0.5, -1.0), (0.5, 0.5, 0.5)), ((0.45, 0.55, 0.5), (0.9, 0.4, 0.6)), ((0.5, 0.5, 4.0), (0.5, 0.5, 9.0))]


@pytest.mark.parametrize("n, n_max, nodes", [(3, 5, (1, 1)), (2000, 150, (2, 256)), (20000, 300, (257, 2000)),
                                             (60000, 8, (9000, 1 << 18)), (400_003, 1, ((1 << 19) + 1, 1 << 21))])
@pytest.mark.parametrize("lam", [None, 0.0, 40.0])
def test_selection_paths_equal_the_oracle(n, n_max, nodes, lam):
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    p = synth.tiny(n, seed=n)
    ot = O.build_tree(p.xyz, p.mass, p.h, seed=1, n_max=n_max)
    t = G.build_lod(*to_dev(p.xyz, p.mass, p.h), n_max=n_max, seed=1)
    assert nodes[0] <= len(ot.nodes) <= nodes[1]
    r, dev = G.Renderer(), torch.device("cuda", 0)
    cams = [synth.look_at(e, c, width=64, height=48, z_near=1e-3) for e, c in CAMS]
    par, orp = G.make_params(lambda_px=lam), O.rparams(lambda_px=lam, n_max=n_max)
    views, want = [], []
    for cam in cams:
        w, st, nd, _ = O.render_lod(ot, cam, orp)
        want.append(w)
        _, acc = r.render(t, cam, par)
        assert st == 0 and r.status() == G.OK and np.array_equal(G.u64(acc), w)
        assert r.stats()["splats"] == nd
        both = sum(r.render_part(t, cam, k, 3, par) for k in range(3))
        assert np.array_equal(G.u64(both), w)
        views.append((t, cam, torch.empty((48, 64), dtype=torch.uint8, device=dev),
                      torch.empty((48, 64), dtype=torch.int64, device=dev)))
    r.reserve_batch(views, par, record_capacity=1 << 24)
    r.render_batch(views, par)
    torch.cuda.synchronize()
    assert r.status() == G.OK
    for (_, _, _, acc), w in zip(views, want):
        assert np.array_equal(G.u64(acc), w)
    t.free()
    r.close()
