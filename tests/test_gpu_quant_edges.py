"""16-bit block codes where a code changes: coordinates on and one ulp beside cell edges, smoothing
lengths and weights on and beside half steps, in root cubes whose code step is and is not a power of
two, one leaf and many nodes, against the oracle bit for bit (the encoder decides most codes in fp32
and must leave these to its FP64 form)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O

from gpu_helpers import same_floats, to_dev

pytestmark = pytest.mark.gpu


def _edge_values(rng, n, lo, step):
    """lo + (c + offset) step for codes c, offset 0 or 1/2, shifted by -1, 0 or 1 ulp (fp32)."""
    c = rng.integers(0, 65536, n) + rng.choice([0.0, 0.5], n)
    c[:6] = np.array([0.0, 0.5, 1.0, 65534.5, 65535.0, 65535.5])[:n]
    v = (lo + c * step).astype(np.float32)
    s = rng.integers(-1, 2, n)
    v = np.where(s < 0, np.nextafter(v, np.float32(-np.inf)), np.where(s > 0, np.nextafter(v, np.float32(np.inf)), v))
    return v.astype(np.float32)


@pytest.mark.parametrize("side,lo", [(1.0, 0.0), (3.0, 0.0), (1.0, -0.3), (7e-3, 0.25)])
@pytest.mark.parametrize("n,n_max", [(5000, 6000), (20000, 300), (1, 5)])
@pytest.mark.parametrize("hstep", [2.0 ** -18, 3.1e-7])
def test_codes_at_their_edges_equal_the_oracle(side, lo, n, n_max, hstep):
    from paper_0811_2055_gb300 import gblod
    torch.cuda.set_device(0)
    rng = np.random.default_rng(int(n + 100 * side))
    xyz = np.stack([_edge_values(rng, n, lo, side / 65536.0) for _ in range(3)], 1)
    h = _edge_values(rng, n, 0.01, hstep)
    mass = _edge_values(rng, n, 1.0, hstep)
    t = gblod.build_lod(*to_dev(xyz, mass, h), n_max=n_max, seed=3, root_lo=(lo, lo, lo), root_side=side).quantize()
    codes, qa, D = O.block_quantize(O.build_tree(xyz, mass, h, seed=3, n_max=n_max, lo=(lo, lo, lo), side=side))
    ex = t.export_block16()
    assert np.array_equal(ex["codes"], codes) and same_floats(ex["qa"], qa)
    for f in ("bmin", "bmax", "h_cull"):
        assert np.array_equal(ex["qnodes"][f], D.nodes[f]), f
    t.free()
