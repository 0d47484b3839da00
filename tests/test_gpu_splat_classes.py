"""The splat kernel's record classes (faint / light / heavy amplitudes, supports below and above 2^15
units, one pair of blocks or both) and its strips, against the oracle bit for bit: amplitudes and
supports on both sides of every class boundary, tiles of one to eight strips with one to four block
rows, image sizes that cut tiles and strips, both radial kernels, in single frames and in a batch."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_0811_2055_gb300 import synth

from gpu_helpers import to_dev

pytestmark = pytest.mark.gpu
D = 1.7  # every point lies in the plane zc = 1.7


def _points(cam, cubic, n=420, seed=5):
    rng = np.random.default_rng(seed)
    W, H, F = cam["width"], cam["height"], cam["f_px"]
    u, v = rng.uniform(-0.5 * W, 1.5 * W, n), rng.uniform(-0.5 * H, 1.5 * H, n)
    sig = np.exp(rng.uniform(np.log(0.4), np.log(900.0), n))
    wq = np.exp2(rng.uniform(8.0, 40.0, n))
    edge = 64.0 if cubic else 128.0 / 3.0  # support of 2^15 units: the narrow / wide boundary
    sig[:40] = edge * (1.0 + rng.uniform(-2e-3, 2e-3, 40))
    sig[40:44] = edge
    wq[44:84] = 2.0 ** rng.choice([22, 23, 31, 32], 40) * (1.0 + rng.uniform(-3e-7, 3e-7, 40))
    wq[84:90] = 2.0 ** 23 - np.arange(6) / 2
    sig[90:130] = rng.uniform(680.0, 690.0, 40)
    sig[130:300] = np.exp(rng.uniform(np.log(1.3), np.log(12.0), 170))  # blobs of a few blocks
    u[130:300], v[130:300] = rng.uniform(-8, W + 8, 170), rng.uniform(-8, H + 8, 170)
    A = 2.0 ** 32 * 10.0 / (7.0 * np.pi) if cubic else 2.0 ** 32 / (2.0 * np.pi * (1.0 - np.exp(-4.5)))
    xyz = np.stack([0.5 - (u - cam["cx"]) * D / F, 0.5 - (v - cam["cy"]) * D / F, np.full(n, 0.5)], 1)
    return (np.ascontiguousarray(xyz, np.float32), (wq * sig * sig / A).astype(np.float32),
            (sig * D / F).astype(np.float32))


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("W,H,tw,th", [(200, 150, 64, 16), (131, 97, 32, 32), (67, 45, 16, 64), (90, 33, 24, 20),
                                       (61, 70, 8, 4), (33, 50, 5, 7), (100, 40, 64, 3)])
def test_record_classes_equal_the_oracle(kernel, W, H, tw, th):
    from paper_0811_2055_gb300 import gblod
    torch.cuda.set_device(0)
    cam = synth.look_at((0.5, 0.5, -1.2), (0.5, 0.5, 0.5), width=W, height=H)
    pts = _points(cam, kernel == 1)
    want, st, nd = O.splat_particles(*pts, cam, O.rparams(kernel=kernel, sigma_min_px=0.3, sigma_max_px=1000.0))
    assert st == 0 and nd > 200
    r = gblod.Renderer()
    par = gblod.make_params(kernel=kernel, sigma_min_px=0.3, sigma_max_px=1000.0, tile_w=tw, tile_h=th,
                            count_updates=True)
    _, acc = r.render_bruteforce(*to_dev(*pts), cam, par)
    assert r.status() == gblod.OK and np.array_equal(gblod.u64(acc), want)
    # the points whose mass an octree takes, as one leaf drawn twice in a batch
    ok = (pts[1] >= 2.0 ** -24) & (pts[1] <= 2.0 ** 24)
    sub = tuple(np.ascontiguousarray(a[ok]) for a in pts)
    assert ok.sum() > 300
    want, st, nd = O.splat_particles(*sub, cam, O.rparams(kernel=kernel, sigma_min_px=0.3, sigma_max_px=1000.0))
    tree = gblod.build_lod(*to_dev(*sub), n_max=len(sub[0]), seed=1)
    views = [(tree, cam, None, torch.empty((H, W), dtype=torch.int64, device="cuda")) for _ in range(2)]
    r.reserve_batch(views, par, record_capacity=1 << 20)
    r.render_batch(views, par)
    assert st == 0 and r.status() == gblod.OK
    for v in views:
        assert np.array_equal(gblod.u64(v[3]), want)
    tree.free()
    r.close()
