"""Views that can only reach the upper levels of a tree select from those alone: eyes inside, on and next to the root
cube, and ever farther away, roots away from the origin, every form of the threshold, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_0811_2055_gb300 import synth

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


# deep trees: 65,000 nodes (flat form), and above 2^19 (level by level unless the view is far)
@pytest.mark.parametrize("n, n_max, lo, side, block16", [(30_000, 1, (0.0, 0.0, 0.0), 1.0, False),
                                                         (30_000, 1, (0.0, 0.0, 0.0), 1.0, True),
                                                         (30_000, 3, (-37.0, 11.5, 1000.0), 0.37, False),
                                                         (30_000, 3, (-37.0, 11.5, 1000.0), 0.37, True),
                                                         (400_003, 1, (0.0, 0.0, 0.0), 1.0, False)])
def test_selection_from_far_and_near(n, n_max, lo, side, block16):
    from paper_0811_2055_gb300 import gblod as G
    torch.cuda.set_device(0)
    p = synth.tiny(n, seed=n_max)
    xyz = (np.asarray(lo) + side * p.xyz.astype(np.float64)).astype(np.float32)
    h = (side * p.h).astype(np.float32)
    ot = O.build_tree(xyz, p.mass, h, seed=1, n_max=n_max, lo=lo, side=side)
    t = G.build_lod(*to_dev(xyz, p.mass, h), n_max=n_max, seed=1, root_lo=lo, root_side=side)
    if block16:
        t.quantize()
        ot = O.block_quantize(ot)[2]
    mid = np.asarray(lo) + 0.5 * side
    fmt = dict(point_format=G.POINTS_BLOCK16) if block16 else {}
    r, dev = G.Renderer(), torch.device("cuda", 0)
    for lam in (None, 0.0, 2.0, 30.0, 1e6, np.inf):
        par, orp = G.make_params(lambda_px=lam, **fmt), O.rparams(lambda_px=lam, n_max=n_max)
        views, want = [], []
        for away in (0.0, 0.5, 0.5 + 1e-12, 0.501, 0.7, 1.5, 4.0, 30.0, 1000.0, 1e5):
            eye = mid + side * np.array([0.13, -0.07, -away]) * (1.0, 1.0, 1.0 if away else 0.0)
            cam = synth.look_at(tuple(eye), tuple(mid if away else mid + (0, 0, side)), width=64, height=48,
                                z_near=1e-3 * side if away < 1e3 else 0.0)
            r.render(t, cam, par, image=None)
            sel = O.select(ot, cam, orp)
            assert np.array_equal(r.last_selection(), sel), (lam, away)
            r.render_part(t, cam, 1, 3, par)
            assert np.array_equal(r.last_selection(), sel[sel % 3 == 1]), (lam, away)
            views.append((t, cam, None, torch.empty((48, 64), dtype=torch.int64, device=dev)))
            want.append(len(sel))
        r.reserve_batch(views, par, record_capacity=1 << 24)
        for some in (views, views[6:], views[:2]):
            r.render_batch(some, par)
            torch.cuda.synchronize()
            got = r.stats()["nodes_selected"]
            assert got == sum(w for v, w in zip(views, want) if any(v is q for q in some)), lam
    r.close()
    t.free()
