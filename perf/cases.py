"""Performance cases: what users of the renderer have it do, through paper_0811_2055_gb300.gblod.

Kinds of a case
---------------
``frame``     one LOD frame of an octree that is already on the device (interactive viewing)
``all``       one frame of every particle, no tree (the full rendering a LOD frame is compared with)
``timestep``  a timestep arrives: its octree is built, its size read, one frame drawn, the octree
              freed; with ``block16`` the points are coded in 16 bits in between
``batch``     several viewers' views of two timesteps in one set of launches (serving)
``fit``       one forward + adjoint step of fitting representatives to images

Particle sets are the recipes of ``synth`` (Plummer spheres; NFW halos + background, optionally one
dominant central halo), drawn on the device so that 150M particles take well under a second.
"""
import math

import numpy as np
import torch

from paper_0811_2055_gb300 import gblod, synth

DEV = "cuda"
MAX_N = 150_000_000  # the data paragraph's particles per timestep


def listed():
    return [
        # the smallest interactive frame: 262,144 particles, 512 x 512 (launch and latency bound)
        dict(name="frame_tiny_512", kind="frame", data="plummer", n=262_144, n_max=16000, width=512, height=512,
             cam="front", at=0.0, kernel=0, block16=False),
        # an ordinary fly-through frame: 16.8M particles at 1080p
        dict(name="frame_mid_1080p", kind="frame", data="halos", n=1 << 24, n_max=16000, width=1920, height=1080,
             cam="helix", at=0.67, kernel=0, block16=False),
        # the paper's timestep, 150M particles, seen from near the central halo: the most pixel work
        dict(name="frame_150m_near", kind="frame", data="central", n=MAX_N, n_max=16000, width=1920, height=1080,
             cam="approach", at=0.43, kernel=0, block16=False),
        # the paper's radial cubic from 16-bit block codes, a ragged window size, a smaller data set
        dict(name="frame_cubic_block16", kind="frame", data="halos", n=3_000_017, n_max=16000, width=1283, height=717,
             cam="helix", at=0.25, kernel=1, block16=True),
        # every particle of the ordinary data set at 1080p
        dict(name="all_mid_1080p", kind="all", data="halos", n=1 << 24, n_max=0, width=1920, height=1080,
             cam="helix", at=0.25, kernel=0, block16=False),
        # every particle of the paper's timestep, the whole box in view: mostly blobs of a few pixels
        dict(name="all_150m_far", kind="all", data="central", n=MAX_N, n_max=0, width=1920, height=1080,
             cam="approach", at=1.0, kernel=0, block16=False),
        # a small timestep with caller ids and unequal masses, previewed in a 640 x 360 window
        dict(name="timestep_1m_ids", kind="timestep", data="halos", n=1_000_003, n_max=2000, width=640, height=360,
             cam="helix", at=0.0, kernel=0, block16=False, ids=True),
        # the ordinary timestep, coded in 16 bits on arrival (fp32 points dropped) and previewed
        dict(name="timestep_mid_block16", kind="timestep", data="halos", n=1 << 24, n_max=16000, width=1280,
             height=720, cam="helix", at=0.0, kernel=0, block16=True, ids=False),
        # the paper's timestep arriving in an interactive session: build + whole-box 1080p frame
        dict(name="timestep_150m", kind="timestep", data="central", n=MAX_N, n_max=16000, width=1920, height=1080,
             cam="approach", at=1.0, kernel=0, block16=False, ids=False),
        # eight viewers at 720p / 1080p / 4K of two timesteps, served as one batch
        dict(name="batch_8_views", kind="batch", data="halos", n=1 << 22, n_max=16000, views=8, cam="orbit", at=0.3,
             kernel=0, block16=False),
        # one step of fitting a node's 16,000 points from eight 128 x 128 views (thousands per octree)
        dict(name="fit_node", kind="fit", n=16_000, views=8, width=128, height=128),
        # one step of fitting a million representatives from 16 views of 256 x 256
        dict(name="fit_1m", kind="fit", n=1 << 20, views=16, width=256, height=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "all", "timestep", "batch", "fit"])
    if kind == "fit":
        w = _log_int(rng, 48, 256)
        return dict(kind=kind, n=_log_int(rng, 4000, 1 << 20), views=rng.randint(1, 16), width=w,
                    height=max(32, int(w * rng.uniform(0.7, 1.0))))
    data = rng.choice(["plummer", "halos", "halos", "central"])
    c = dict(kind=kind, data=data, n=_log_int(rng, 1 << 17, 1 << 24), kernel=rng.choice([0, 0, 1]), at=rng.random(),
             cam={"plummer": "front", "halos": "helix", "central": "approach"}[data], block16=False,
             n_max=0 if kind == "all" else rng.choice([16000, 16000, 2000, 500]))
    if kind == "batch":
        return dict(c, cam="orbit", n=_log_int(rng, 1 << 17, 1 << 22), views=rng.randint(2, 10))
    w = _log_int(rng, 256, 2200)
    c.update(width=w, height=max(144, int(w * rng.uniform(0.5, 0.65))))
    if kind == "frame":
        c["block16"] = rng.random() < 0.3
    if kind == "timestep":
        c.update(block16=rng.random() < 0.3, ids=rng.random() < 0.4)
    return c


# ----------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV)


def _isotropic(g, n):
    z = 2.0 * _rand(g, n) - 1.0
    phi = (2.0 * math.pi) * _rand(g, n)
    s = torch.sqrt(torch.clamp(1.0 - z * z, min=0.0))
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), z], 1)


def _wrap(p):
    return torch.clamp(p - torch.floor(p), 0.0, float(synth.ONE_MINUS))


def _plummer(n, seed):
    """80% in 64 Plummer spheres, 20% background; h = 0.002 exp(Z / 2)."""
    g = _gen(seed)
    n_cl = (4 * n) // 5
    a = torch.exp(math.log(0.005) + math.log(10.0) * _rand(g, 64))
    centres = _rand(g, 64, 3)
    sph = torch.arange(n_cl, device=DEV) % 64
    u = torch.clamp(_rand(g, n_cl), min=1e-7)
    r = torch.clamp(a[sph] / torch.sqrt(torch.clamp(u ** (-2.0 / 3.0) - 1.0, min=1e-12)), max=0.5)
    pos = torch.cat([centres[sph] + r[:, None] * _isotropic(g, n_cl), _rand(g, n - n_cl, 3)])
    h = 0.002 * torch.exp(0.5 * torch.randn(n, generator=g, device=DEV))
    perm = torch.randperm(n, generator=g, device=DEV)
    return _wrap(pos[perm]).contiguous(), h.contiguous()


def _halos(n, seed, central):
    """NFW halos (dN/dM ~ M^-1.9 over three decades) + 10% background, optionally a central halo
    holding 30%; h = 1.2 x the local mean spacing of the host halo's profile."""
    g = _gen(seed)
    rng = np.random.default_rng(int(seed))
    n_halos = max(1, round((65536 / 150e6 if central else 4096 / (1 << 24)) * n))
    n_bg, n_c = round(0.10 * n), round(0.30 * n) if central else 0
    gm = 1.0 - 1.9
    m = (1.0 + rng.random(n_halos) * (1000.0 ** gm - 1.0)) ** (1.0 / gm)
    edges = np.floor(np.concatenate([[0.0], np.cumsum(m)]) / m.sum() * (n - n_bg - n_c)).astype(np.int64)
    edges[-1] = n - n_bg - n_c
    cnt, conc, rvir = np.diff(edges), rng.uniform(5.0, 15.0, n_halos), 0.05 * (m / 1000.0) ** (1.0 / 3.0)
    centres = rng.random((n_halos, 3))
    if central:
        cnt, conc, rvir = np.append(cnt, n_c), np.append(conc, 10.0), np.append(rvir, 0.25)
        centres = np.concatenate([centres, [[0.5, 0.5, 0.5]]])
    bucket = np.clip(((conc - 5.0) / 10.0 * 64).astype(np.int64), 0, 63)
    c64 = 5.0 + 10.0 * (np.arange(64) + 0.5) / 64
    mu = lambda x: np.log1p(x) - x / (1.0 + x)  # noqa: E731
    grid = np.linspace(0.0, 1.0, 4097)
    inv = np.stack([np.interp(np.linspace(0.0, 1.0, 4097), mu(c * grid) / mu(c), grid) for c in c64])
    cu = c64[bucket]
    rs = rvir / cu
    rho = cnt / (4.0 * np.pi * rs ** 3 * mu(cu))
    up = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV)  # noqa: E731
    n_h = n - n_bg
    host = torch.repeat_interleave(torch.arange(len(cnt), device=DEV), torch.from_numpy(cnt).to(DEV), output_size=n_h)
    t = _rand(g, n_h) * 4096.0
    k = torch.clamp(t.long(), max=4095)
    f = t - k
    k += torch.from_numpy(bucket * 4097).to(DEV)[host]
    table = up(inv).reshape(-1)
    x = (table[k] * (1.0 - f) + table[k + 1] * f) * up(cu)[host]
    del t, k, f
    pos = torch.empty(n, 3, device=DEV)
    pos[:n_h] = up(centres)[host] + (x * up(rs)[host])[:, None] * _isotropic(g, n_h)
    pos[n_h:] = _rand(g, n_bg, 3)
    x = torch.clamp(x, min=1e-6)
    h = torch.empty(n, device=DEV)
    h[:n_h] = torch.clamp(1.2 * (up(rho)[host] / (x * (1.0 + x) ** 2)) ** (-1.0 / 3.0), 1e-5, 0.02)
    h[n_h:] = 1.2 * max(n_bg, 1) ** (-1.0 / 3.0)
    del host, x
    perm = torch.randperm(n, generator=g, device=DEV)
    return _wrap(pos[perm]).contiguous(), h[perm].contiguous()


def _particles(case, seed):
    xyz, h = _plummer(case["n"], seed) if case["data"] == "plummer" else _halos(case["n"], seed,
                                                                               case["data"] == "central")
    mass = torch.ones(case["n"], device=DEV)
    return xyz, mass, h


def _camera(case, seed, width, height, at):
    jitter = 1e-3 * (seed % 97)  # another seed is another moment of the same path
    if case["cam"] == "front":
        return synth.look_at((0.5 + jitter, 0.5, -1.0 + at), (0.5, 0.5, 0.5), width=width, height=height)
    if case["cam"] == "helix":
        return synth.helix_view(239.0 * at + 10 * jitter, width=width, height=height)
    if case["cam"] == "approach":  # 0.01 to 1.5 box sides from the central halo
        d = 0.01 * 150.0 ** at * (1.0 + jitter)
        return synth.look_at((0.5, 0.5, 0.5 - d), (0.5, 0.5, 0.5), width=width, height=height, z_near=1e-4)
    a = 2.0 * math.pi * (at + jitter)
    r = 0.6 + 0.8 * ((7.0 * at) % 1.0)
    return synth.look_at((0.5 + r * math.cos(a), 0.6, 0.5 + r * math.sin(a)), (0.5, 0.5, 0.5), width=width,
                         height=height)


def _params(case):
    return gblod.make_params(kernel=case["kernel"],
                             point_format=gblod.POINTS_BLOCK16 if case["block16"] else gblod.POINTS_FLOAT)


VIEW_SIZES = ((1280, 720), (1920, 1080), (1280, 720), (3840, 2160), (1280, 720), (1920, 1080))


def _view_sizes(case):
    return [VIEW_SIZES[i % len(VIEW_SIZES)] for i in range(case["views"])]


def prepare(case, seed):
    kind = case["kind"]
    r = gblod.Renderer()
    if kind == "fit":
        g = _gen(seed)
        n, nv = case["n"], case["views"]
        xyz, h = _halos(n, seed, False)
        logh = torch.log(h)
        w = 16.0 * (0.5 + _rand(g, n))
        grad = torch.randn(nv, case["height"], case["width"], generator=g, device=DEV)
        gold = math.pi * (3.0 - math.sqrt(5.0))
        cams = []
        for k in range(nv):
            y = 1.0 - 2.0 * (k + 0.5) / nv
            s = 1.5 * math.sqrt(max(0.0, 1.0 - y * y))
            eye = (0.5 + s * math.cos(gold * k), 0.5 + 1.5 * y, 0.5 + s * math.sin(gold * k))
            cams.append(synth.look_at(eye, (0.5, 0.5, 0.5), width=case["width"], height=case["height"]))
        leaf = [t.requires_grad_(True) for t in (xyz, w, logh)]
        return dict(kind=kind, r=r, leaf=leaf, grad=grad, cams=cams, params=gblod.make_params())
    xyz, mass, h = _particles(case, seed)
    st = dict(kind=kind, r=r, params=_params(case), n_max=case["n_max"], seed=seed, block16=case["block16"])
    if kind == "batch":
        st["trees"] = [gblod.build_lod(xyz, mass, h, n_max=case["n_max"], seed=seed)]
        moved = _wrap(xyz + 0.002 * torch.sin(40.0 * xyz.flip(1))).contiguous()
        st["trees"].append(gblod.build_lod(moved, mass, h, n_max=case["n_max"], seed=seed))
        st["views"] = []
        for i, (w, hh) in enumerate(_view_sizes(case)):
            cam = _camera(case, seed, w, hh, (case["at"] + 0.37 * i) % 1.0)
            st["views"].append((st["trees"][i % 2], cam, torch.empty(hh, w, dtype=torch.uint8, device=DEV),
                                torch.empty(hh, w, dtype=torch.int64, device=DEV)))
        r.reserve_batch(st["views"], st["params"], record_capacity=1 << 29)
        return st
    st["cam"] = _camera(case, seed, case["width"], case["height"], case["at"])
    if kind == "frame":
        st["tree"] = gblod.build_lod(xyz, mass, h, n_max=case["n_max"], seed=seed)
        if case["block16"]:
            st["tree"].quantize(drop_float=True)
        return st
    st["ids"] = None
    if case.get("ids"):
        g = _gen(seed + 1)
        st["ids"] = torch.randperm(case["n"], generator=g, device=DEV).int()
        mass = torch.exp(0.3 * torch.randn(case["n"], generator=g, device=DEV))
    st["parts"] = (xyz, mass, h)
    return st


# ----------------------------------------------------------------------------- one pass
def run(st):
    kind, r = st["kind"], st["r"]
    if kind == "frame":
        return r.render(st["tree"], st["cam"], st["params"])
    if kind == "all":
        return r.render_bruteforce(*st["parts"], st["cam"], st["params"])
    if kind == "timestep":
        tree = gblod.build_lod(*st["parts"], ids=st["ids"], n_max=st["n_max"], seed=st["seed"])
        info = tree.info()
        if st["block16"]:
            tree.quantize(drop_float=True)
        img, acc = r.render(tree, st["cam"], st["params"])
        tree.free()
        return [int(info.n_nodes), int(info.n_points), int(info.depth_max), int(info.equal_mass)], img, acc
    if kind == "batch":
        r.render_batch(st["views"], st["params"])
        return [(v[2], v[3]) for v in st["views"]]
    img = gblod.SplatImages.apply(*st["leaf"], st["cams"], r, st["params"])
    return img.detach(), torch.autograd.grad(img, st["leaf"], st["grad"])


def work(case):
    if case["kind"] == "fit":
        px = case["views"] * case["width"] * case["height"]
        # points read for both directions and gradients written once; images written, gradients read;
        # per (view, point) projection and its chain rule (about 60 operations)
        return {"bytes": 2 * 20.0 * case["n"] + 20.0 * case["n"] + 8.0 * px, "flops": 60.0 * case["n"] * case["views"]}
    if case["kind"] == "batch":
        px = sum(w * h for w, h in _view_sizes(case))
        return {"bytes": 9.0 * px + 2 * min(20.0 * case["n"], 20.0 * 10 * px)}
    px = case["width"] * case["height"]
    drawn = (10.0 if case["block16"] else 20.0) * min(case["n"], 10 * px)  # about ten points a pixel (depth paragraph)
    if case["kind"] == "frame":
        return {"bytes": 9.0 * px + drawn}
    if case["kind"] == "all":
        return {"bytes": 9.0 * px + 20.0 * case["n"]}
    # octree: particles in, sorted keys + permutation + about 1.6 stored points a particle out
    return {"bytes": 9.0 * px + drawn + (20.0 + 12.0 + 1.6 * 24.0) * case["n"]}


# ----------------------------------------------------------------------------- 64-bit values
def exact(case, seed):
    """Frames are whole numbers.  The float splat and its gradients: the formulas in 64 bits."""
    if case["kind"] != "fit":
        return None
    st = prepare(case, seed)
    xyz, w, logh = (t.detach().double() for t in st["leaf"])
    W, H, par = case["width"], case["height"], st["params"]
    img = torch.zeros(case["views"], H, W, dtype=torch.float64, device=DEV)
    gx, gw, gl = torch.zeros_like(xyz), torch.zeros_like(w), torch.zeros_like(logh)
    cut = math.exp(-4.5)
    norm = 1.0 / (2.0 * math.pi * (1.0 - 5.5 * cut))
    for v, cam in enumerate(st["cams"]):
        R = torch.tensor([cam["right"], cam["up"], cam["fwd"]], dtype=torch.float64, device=DEV)
        F = cam["f_px"]
        c = (xyz - torch.tensor(cam["eye"], dtype=torch.float64, device=DEV)) @ R.T
        iz = 1.0 / c[:, 2]
        u, t = cam["cx"] + F * c[:, 0] * iz, cam["cy"] - F * c[:, 1] * iz
        raw = F * torch.exp(logh) * iz
        s = torch.clamp(raw, par.sigma_min_px, par.sigma_max_px)
        free = ((raw >= par.sigma_min_px) & (raw <= par.sigma_max_px)).double()
        reach = 3.0 * s + 1.0
        seen = (c[:, 2] > cam["z_near"]) & (u + reach >= 0) & (u - reach <= W) & (t + reach >= 0) & (t - reach <= H)
        flat, upstream = img[v].reshape(-1), st["grad"][v].double().reshape(-1)
        half, lo = 3, 0.0
        while lo < float(reach.max()):
            idx = torch.nonzero(seen & (reach > lo) & (reach <= half)).reshape(-1)
            side = 2 * half + 1
            step = max(1, (1 << 24) // (side * side))
            off = torch.arange(-half, half + 1, device=DEV)
            for b in range(0, idx.numel(), step):
                i = idx[b:b + step]
                ui, ti, si, wi = u[i, None], t[i, None], s[i, None], w[i, None]
                x, y = torch.floor(ui).long() + off, torch.floor(ti).long() + off
                inx, iny = (x >= 0) & (x < W), (y >= 0) & (y < H)
                dx, dy = (x + 0.5 - ui)[:, None, :], (y + 0.5 - ti)[:, :, None]
                r2, s3 = dx * dx + dy * dy, si[:, :, None]
                ok = (r2 < 9.0 * s3 * s3) & inx[:, None, :] & iny[:, :, None]
                pix = torch.where(ok, y[:, :, None] * W + x[:, None, :], 0)
                e = torch.where(ok, torch.exp(-r2 / (2.0 * s3 * s3)), 0.0) * (norm / (s3 * s3))
                k = torch.where(ok, e - cut * norm / (s3 * s3), 0.0)
                flat.index_add_(0, pix.reshape(-1), (wi[:, :, None] * k).reshape(-1))
                gi = torch.where(ok, upstream[pix], 0.0)
                tw = (gi * k).sum((1, 2))
                gi = gi * wi[:, :, None]
                tu = (gi * e * dx / (s3 * s3)).sum((1, 2))
                tv = (gi * e * dy / (s3 * s3)).sum((1, 2))
                ts = (gi * (e * r2 / s3 ** 3 - 2.0 * k / s3)).sum((1, 2))
                ci, zi = c[i], iz[i]
                dz = (-tu * F * ci[:, 0] + tv * F * ci[:, 1]) * zi * zi - ts * free[i] * s[i] * zi
                gx.index_add_(0, i, torch.stack([tu * F * zi, -tv * F * zi, dz], 1) @ R)
                gw.index_add_(0, i, tw)
                gl.index_add_(0, i, ts * free[i] * s[i])
            lo, half = float(half), 2 * half
    return img, (gx, gw, gl)
