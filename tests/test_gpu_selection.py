"""Representatives of unequal masses, whose keys are binned in fp32 and compared in FP64 only near the
threshold, and of equal masses at the bin counts' edges: node counts around 64, 4096 and the chunk, masses from
equal but one to sixty orders of two apart, thresholds from 1 to all but one particle, against the oracle bit
for bit, with the codes kept (the library's pool) and computed twice (a caller's allocator)."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import oracle as O

from gpu_helpers import compare_trees, to_dev
from test_gpu_alloc_failure import Budget

pytestmark = pytest.mark.gpu


def _mass(kind, n, rng):
    if kind == "equal":
        return np.full(n, 3.0)
    if kind == "one":       # equal but one: every key near its node's expected threshold
        m = np.full(n, 3.0)
        m[n // 2] = 1e6
        return m
    if kind == "tiny":      # the smallest allowed
        return 2.0 ** -24 * rng.uniform(1.0, 3.0, n)
    if kind == "two":       # a few hold nearly all the mass: a threshold far above the expected one
        return np.where(rng.uniform(0.0, 1.0, n) < 0.05, 1e7, 1e-7)
    return np.exp2(rng.uniform(-24.0, 24.0, n)) # "wide"


@pytest.mark.parametrize("kind", ["equal", "one", "tiny", "two", "wide"])
@pytest.mark.parametrize("n, n_max", [(63, 62), (64, 1), (65, 20), (4095, 4094), (4097, 1000), (8193, 4096),
                                      (50001, 300), (50001, 49999)])
def test_selection_equals_the_oracle(kind, n, n_max):
    from paper_0811_2055_gb300 import gblod
    torch.cuda.set_device(0)
    rng = np.random.default_rng(n + n_max)
    xyz = rng.uniform(0.0, 1.0, (n, 3)).astype(np.float32)
    h = rng.uniform(1e-4, 1e-2, n).astype(np.float32)
    mass = _mass(kind, n, rng).astype(np.float32)
    ot = O.build_tree(xyz, mass, h, seed=n, n_max=n_max)
    d = to_dev(xyz, mass, h)
    t = gblod.build_lod(*d, n_max=n_max, seed=n)
    compare_trees(t.export(), ot)
    t.free()
    bp, out, b = gblod.BuildParams(), C.c_void_p(), Budget(1 << 40)
    bp.seed, bp.n_max, bp.root_side = n, n_max, 1.0
    assert gblod.lib().gblod_build_lod(d[0].data_ptr(), d[1].data_ptr(), d[2].data_ptr(), None, n, C.byref(bp),
                                       C.byref(b.hook()), torch.cuda.current_stream().cuda_stream,
                                       C.byref(out)) == gblod.OK
    t = gblod.Octree(out.value)
    compare_trees(t.export(), ot)
    t.free()
    torch.cuda.synchronize()
    assert b.used == 0
