"""Octree builds at the sizes where their kernels have edges: particle counts around the sort's tile and
the selection's chunk, keys with few varying digits (odd and even numbers of sort passes), coincident
particles and one dense clump, equal and unequal masses, caller ids, and both ways the work arrays are
allocated (the library's pool; a caller's allocator), against the oracle bit for bit."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import oracle as O

from gpu_helpers import compare_trees, to_dev
from test_gpu_alloc_failure import Budget

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 31, 33, 4095, 4096, 4097, 8192, 12289, 40000]
KINDS = ["uniform", "corner", "line", "coincident", "clump"]


def _data(kind, n, seed):
    rng = np.random.default_rng(seed)
    xyz = rng.uniform(0.0, 1.0, (n, 3))
    if kind == "corner":    # the top key digits are the same for all
        xyz *= 2.0 ** -9
    elif kind == "line":    # one axis varies
        xyz[:, 1:] = 0.375
    elif kind == "coincident":
        xyz[n // 3:] = xyz[0]
    elif kind == "clump":   # most of the particles share the first 15 levels
        xyz[: 3 * n // 4] = 0.3 + xyz[: 3 * n // 4] * 2.0 ** -15
    mass = np.exp(rng.normal(0.0, 2.0, n)) if seed % 2 else np.full(n, 0.75)
    h = rng.uniform(1e-4, 1e-2, n)
    ids = rng.permutation(max(4 * n, 8))[:n].astype(np.int32) if seed % 3 == 0 else None
    return [a.astype(np.float32) for a in (xyz, mass, h)] + [ids]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", KINDS)
def test_build_edges_equal_the_oracle(kind, n):
    from paper_0811_2055_gb300 import gblod
    torch.cuda.set_device(0)
    for seed, n_max in ((n % 7 + 1, 24), (n % 5 + 2, 700), (3, 1)):
        if n_max == 1 and n > 5000:
            continue
        xyz, mass, h, ids = _data(kind, n, seed)
        ot = O.build_tree(xyz, mass, h, ids=ids, seed=seed, n_max=n_max)
        d = to_dev(xyz, mass, h)
        dids = None if ids is None else torch.from_numpy(ids).cuda()
        t = gblod.build_lod(*d, ids=dids, n_max=n_max, seed=seed)
        compare_trees(t.export(), ot)
        t.free()
        # the same build with the work arrays from a caller's allocator
        bp, out, b = gblod.BuildParams(), C.c_void_p(), Budget(1 << 40)
        bp.seed, bp.n_max, bp.root_side = seed, n_max, 1.0
        st = gblod.lib().gblod_build_lod(d[0].data_ptr(), d[1].data_ptr(), d[2].data_ptr(),
                                         None if dids is None else dids.data_ptr(), n, C.byref(bp),
                                         C.byref(b.hook()), torch.cuda.current_stream().cuda_stream, C.byref(out))
        assert st == gblod.OK
        t = gblod.Octree(out.value)
        compare_trees(t.export(), ot)
        t.free()
        torch.cuda.synchronize()
        assert b.used == 0


@pytest.mark.parametrize("n, n_max", [(2, 1), (4096, 1), (4097, 4096), (8193, 1), (30000, 2), (9000, 8999), (9000, 9000)])
@pytest.mark.parametrize("kind", KINDS + ["pairs"])
def test_refined_nodes_equal_the_oracle(kind, n, n_max):
    """Node tables at the edges of the pass that finds the refined nodes: blocks of 4096 positions full of
    them, none, chains of single children down to the last level, runs of equal keys that end a block."""
    from paper_0811_2055_gb300 import gblod
    torch.cuda.set_device(0)
    xyz, mass, h, _ = _data("uniform" if kind == "pairs" else kind, n, 4)
    if kind == "pairs":     # every particle twice: over-full nodes at the last level
        xyz[1::2] = xyz[: len(xyz[1::2]) * 2: 2]
    ot = O.build_tree(xyz, mass, h, seed=4, n_max=n_max)
    t = gblod.build_lod(*to_dev(xyz, mass, h), n_max=n_max, seed=4)
    compare_trees(t.export(), ot)
    t.quantize()
    qn, on = t.export_block16()["qnodes"], O.block_quantize(ot)[2].nodes
    for f in ("bmin", "bmax", "h_cull", "parent"):
        assert np.array_equal(qn[f], on[f]), f
    t.free()
