"""Performance cases of the compositional sparse-voxel renderer: what users of the library have it do.

A case is a dict of plain values.  Its "kind" says which entry points a pass goes through:

* ``grid_train``   forward and backward through ``torch.autograd`` of one uniform grid (the plain method);
* ``train``        forward and backward of a street scene: a LiDAR-shaped background octree and posed actors;
* ``render``       forward only, no state kept;
* ``lift``         the weights export of a saved render, a feature render and a fusion over it;
* ``features``     a feature render and a fusion over slot lists a program exported earlier and kept;
* ``init``         LiDAR-guided initialisation of a leaf set;
* ``sky``          the sky composite and its backward;
* ``serve``        a burst of requests of mixed resolution through the render server.

Scenes are made on the GPU from the seed: the shapes (leaf counts, levels, actors, cameras, densities, SH
coefficients) are those of the repository's generators in ``synth``.  ``work`` counts each input read once and
each output written once; FLOPs are the ray-box tests and segments of the rendering equation at the segment
counts these scenes have (about 17 per pixel on a street, 11 on the grid).
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2606_23031_gb300 as dv

DEV = "cuda"
SH_C0 = 0.28209479177387814
V_FAR, V_CLOSE = -10.0, -2.0


# ---------------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: one 64x64 view of a 16^3 grid with degree-0 colours, a training step
        {"name": "grid64_train", "kind": "grid_train", "level": 4, "W": 64, "H": 64, "K": 1},
        # one serving request alone: a small view of a street with 20 actors, forward only
        {"name": "view480_render", "kind": "render", "leaves": 500_000, "actors": 20, "cells": 20_000, "sh": 3,
         "cams": 1, "W": 480, "H": 270, "K": 1},
        # novel-view rendering of the benchmark's frame
        {"name": "street1080_render", "kind": "render", "leaves": 500_000, "actors": 3, "cells": 20_000, "sh": 3,
         "cams": 1, "W": 1920, "H": 1080, "K": 1},
        # the benchmark's training step through autograd
        {"name": "street1080_train", "kind": "train", "leaves": 500_000, "actors": 3, "cells": 20_000, "sh": 3,
         "cams": 1, "W": 1920, "H": 1080, "K": 1, "normals": False, "shared": False},
        # the other options in one step: an odd image size, normals, four samples per segment, degree-2
        # colours (rows of 27 floats), densities that live on shared grid corners
        {"name": "odd957_train", "kind": "train", "leaves": 200_000, "actors": 5, "cells": 20_000, "sh": 2,
         "cams": 1, "W": 957, "H": 541, "K": 4, "normals": True, "shared": True},
        # a training step on a large scene: six surround cameras in one call
        {"name": "surround8m_train", "kind": "train", "leaves": 8_000_000, "actors": 20, "cells": 40_000, "sh": 3,
         "cams": 6, "W": 1920, "H": 1080, "K": 1, "normals": False, "shared": False},
        # the largest scene: 32M leaves, 64 actors, two 4K cameras, forward only
        {"name": "stress4k_render", "kind": "render", "leaves": 32_000_000, "actors": 64, "cells": 40_000, "sh": 3,
         "cams": 2, "W": 3840, "H": 2160, "K": 1},
        # 2-D features lifted into the voxels right after a render, a channel count that is no power of two
        {"name": "lift960_c40", "kind": "lift", "leaves": 500_000, "actors": 3, "cells": 20_000, "sh": 1,
         "cams": 1, "W": 960, "H": 540, "K": 1, "channels": 40},
        # feature training over weights exported once: 64 channels on a full frame
        {"name": "features1080_c64", "kind": "features", "W": 1920, "H": 1080, "slots": 17, "channels": 64},
        # one initialisation round of the benchmark's background from its LiDAR sweep
        {"name": "init500k", "kind": "init", "leaves": 500_000, "cams": 6, "W": 1920, "H": 1080},
        # the sky epilogue of a training step, the benchmark's environment map
        {"name": "sky1080", "kind": "sky", "cams": 1, "W": 1920, "H": 1080, "He": 1024, "We": 2048},
        # continuous batching: requests of three resolutions that queue up while admission is held
        {"name": "serve24", "kind": "serve", "leaves": 500_000, "actors": 20, "cells": 20_000, "sh": 3,
         "requests": 24, "max_views": 16, "workers": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid_train", "train", "train", "train", "render", "render", "lift", "features", "init", "sky",
                       "serve"])
    W = _log(rng, 320, 1920)
    H = max(32, int(W * rng.uniform(0.4, 0.8)))
    if kind == "grid_train":
        return {"kind": kind, "level": rng.choice([3, 4, 5]), "W": _log(rng, 24, 128), "H": _log(rng, 24, 128),
                "K": rng.choice([1, 1, 2, 3])}
    scene = {"leaves": _log(rng, 30_000, 4_000_000), "actors": rng.choice([0, 1, 3, 8, 20]),
             "cells": _log(rng, 5_000, 40_000), "sh": rng.choice([0, 1, 2, 3, 3, 3])}
    if kind == "train":
        scene["actors"] = min(scene["actors"], 20)
        return {"kind": kind, **scene, "cams": rng.choice([1, 1, 2, 3]), "W": W, "H": H, "K": rng.choice([1, 1, 1, 2, 4]),
                "normals": rng.random() < 0.3, "shared": rng.random() < 0.3}
    if kind == "render":
        W = _log(rng, 320, 3840)
        return {"kind": kind, **scene, "cams": rng.choice([1, 1, 2, 4]), "W": W, "H": max(32, int(W * rng.uniform(0.4, 0.7))),
                "K": rng.choice([1, 1, 1, 2])}
    if kind == "lift":
        return {"kind": kind, **scene, "cams": 1, "W": W, "H": H, "K": 1, "channels": rng.choice([3, 8, 16, 19, 40, 64, 100])}
    if kind == "features":
        return {"kind": kind, "W": W, "H": H, "slots": rng.randint(8, 30),
                "channels": rng.choice([1, 4, 8, 16, 19, 32, 40, 64, 100, 128])}
    if kind == "init":
        return {"kind": kind, "leaves": _log(rng, 30_000, 1_000_000), "cams": rng.choice([1, 3, 6, 12]), "W": W, "H": H}
    if kind == "sky":
        We = _log(rng, 64, 4096)
        return {"kind": kind, "cams": rng.choice([1, 2, 6]), "W": W, "H": H, "He": max(16, We // 2 + rng.randint(-3, 3)), "We": We}
    scene["leaves"] = _log(rng, 30_000, 1_000_000)
    return {"kind": kind, **scene, "requests": rng.randint(4, 32), "max_views": rng.choice([4, 8, 16]),
            "workers": rng.choice([1, 2, 3])}


# ---------------------------------------------------------------------------------------------------
# scenes (made on the GPU from the seed)
# ---------------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _pose(R, t):
    return SimpleNamespace(R=np.asarray(R, np.float32).reshape(3, 3), t=np.asarray(t, np.float32).reshape(3))


def _identity():
    return _pose(np.eye(3), np.zeros(3))


def _rot_z(a):
    c, s = math.cos(a), math.sin(a)
    return np.array([[c, -s, 0.0], [s, c, 0.0], [0.0, 0.0, 1.0]])


def _look(eye, target):
    eye, f = np.asarray(eye, np.float64), np.asarray(target, np.float64) - np.asarray(eye, np.float64)
    f /= np.linalg.norm(f)
    r = np.cross(f, [0.0, 0.0, 1.0])
    r /= np.linalg.norm(r)
    return _pose(np.stack([r, np.cross(f, r), f], 1), eye)


def _camera(W, H, pose, near, far, fov=60.0):
    fx = float(np.float32(W / 2.0 / math.tan(math.radians(fov) / 2.0)))
    return SimpleNamespace(W=int(W), H=int(H), fx=fx, fy=fx, cx=W / 2.0, cy=H / 2.0, pose=pose, near=near, far=far)


def _vehicle_camera(W, H, yaw, position, far=400.0):
    p = np.asarray(position, np.float64)
    return _camera(W, H, _look(p, p + np.array([math.cos(yaw), math.sin(yaw), 0.0])), 0.1, far)


def _pack(level, i, j, k):
    return (level << 57) | (k << 38) | (j << 19) | i


_OFF = [[c & 1, (c >> 1) & 1, (c >> 2) & 1] for c in range(8)]


def _box_distance(p, c, h):
    q = (p - c).abs() - h
    out = q.clamp(min=0).square().sum(-1).sqrt()
    return (out + q.amax(-1).clamp(max=0)).abs()


def _extent(leaves):
    """Levels and extents of a LiDAR-shaped background of about that many leaves."""
    if leaves > 12_000_000:
        return SimpleNamespace(root=500.0, cz=20.0, half=250.0, height=40.0, lmin=6, lmax=16, fine=4.0, ground=1.25, wall=0.5)
    lmax = 10 if leaves < 100_000 else 12 if leaves <= 1_000_000 else 14
    per = (2.0, 0.8) if lmax <= 12 else (1.5, 0.625)
    return SimpleNamespace(root=200.0, cz=15.0, half=100.0, height=30.0, lmin=6, lmax=lmax, fine=6.0, ground=per[0], wall=per[1])


def _buildings(rng, e, n=20):
    """Axis-aligned boxes off the road corridor along x."""
    cs, hs = [], []
    for _ in range(10000):
        if len(cs) == n:
            break
        size = np.array([rng.uniform(5, 30), rng.uniform(5, 30), min(rng.uniform(5, 30), e.height - 1.0)])
        c = np.array([rng.uniform(-e.half + size[0] / 2, e.half - size[0] / 2),
                      rng.uniform(-e.half + size[1] / 2, e.half - size[1] / 2), size[2] / 2])
        if abs(c[1]) - size[1] / 2 < 12.0:
            continue
        if all(np.any(np.abs(c - c2) > size / 2 + h2 + 1.0) for c2, h2 in zip(cs, hs)):
            cs.append(c)
            hs.append(size / 2)
    return np.array(cs), np.array(hs)


def _sweep(e, leaves, bc, bh, g):
    """LiDAR-like points [m, 3]: ground hits ~ 1/r^2 around the sensor, building faces by area / distance^2."""
    ng, nw = int(e.ground * leaves), int(e.wall * leaves)
    r = 1.5 * (e.half * math.sqrt(2.0) / 1.5) ** torch.rand(ng, device=DEV, generator=g)
    a = 2 * math.pi * torch.rand(ng, device=DEV, generator=g)
    ground = torch.stack([r * a.cos(), r * a.sin(), torch.zeros_like(r)], 1)
    ground = ground[(ground[:, :2].abs() < e.half).all(1)]
    centre, span, weight = [], [], []
    for c, h in zip(bc, bh):
        for ax, sgn in ((0, -1), (0, 1), (1, -1), (1, 1), (2, 1)):
            fc, hv = c.copy(), h.copy()
            fc[ax] += sgn * h[ax]
            hv[ax] = 0.0
            u, v = [x for x in range(3) if x != ax]
            centre.append(fc)
            span.append(hv)
            weight.append(4 * h[u] * h[v] / max(float(fc @ fc), 25.0))
    centre, span = (torch.tensor(np.array(x), dtype=torch.float32, device=DEV) for x in (centre, span))
    f = torch.multinomial(torch.tensor(weight, device=DEV), nw, replacement=True, generator=g)
    wall = centre[f] + (2 * torch.rand(nw, 3, device=DEV, generator=g) - 1) * span[f]
    p = torch.cat([ground, wall])
    return p + 0.05 * torch.randn(p.shape, device=DEV, generator=g)


def _member(x, table):
    if not table.numel():
        return torch.zeros_like(x, dtype=torch.bool)
    return table[torch.searchsorted(table, x).clamp(max=table.numel() - 1)] == x


def _leaf_set(e, pts, lo):
    """Leaf keys of a coarse grid split where points fall, and whether each leaf holds a point."""
    cell = torch.floor((pts - lo) * ((1 << e.lmax) / e.root)).long()
    cell = cell[((cell >= 0) & (cell < (1 << e.lmax))).all(1)]
    code = lambda c: (c[:, 2] << 42) | (c[:, 1] << 21) | c[:, 0]
    occ = {e.lmax: torch.unique(code(cell))}
    del cell
    for lv in range(e.lmax - 1, e.lmin - 1, -1):
        occ[lv] = torch.unique((occ[lv + 1] >> 1) & ~((1 << 20) | (1 << 41)))
    s0, n0 = e.root / (1 << e.lmin), 1 << e.lmin
    ax = torch.arange(n0, device=DEV)
    mid = (ax + 0.5) * s0
    keep = [ax[(mid + float(lo[0])).abs() < e.half], ax[(mid + float(lo[1])).abs() < e.half],
            ax[(mid + float(lo[2]) > -s0) & (mid + float(lo[2]) < e.height + s0)]]
    cur = torch.cartesian_prod(*keep)
    off = torch.tensor(_OFF, device=DEV)
    edges = torch.tensor([(e.fine * 2.0 ** t) ** 2 for t in range(e.lmax - e.lmin + 1)], device=DEV)
    keys, hits = [], []
    for lv in range(e.lmin, e.lmax + 1):
        is_occ = _member(code(cur), occ[lv])
        split = torch.zeros_like(is_occ)
        if lv < e.lmax:
            r2 = ((cur[:, :2] + 0.5) * (e.root / (1 << lv)) + lo[:2]).square().sum(1)
            split = is_occ & (lv < (e.lmax - torch.searchsorted(edges, r2, right=True)).clamp(min=e.lmin))
        leaf = cur[~split]
        keys.append(_pack(lv, leaf[:, 0], leaf[:, 1], leaf[:, 2]))
        hits.append(is_occ[~split])
        cur = (2 * cur[split][:, None, :] + off).reshape(-1, 3)
        if not cur.numel():
            break
    return torch.cat(keys), torch.cat(hits)


def _background(leaves, sh, seed):
    """LiDAR-shaped background octree: a coarse grid split where points fall, finer near the sensor, trimmed to
    ``leaves`` (empty space first), densities falling off from the nearest surface."""
    e, rng, g = _extent(leaves), random.Random(seed), _gen(seed)
    bc, bh = _buildings(rng, e)
    lo = torch.tensor([-e.root / 2, -e.root / 2, e.cz - e.root / 2], device=DEV)
    off = torch.tensor(_OFF, device=DEV)
    for more in (1, 2, 4, 8):  # a denser sweep where this one gives too few leaves
        pts = _sweep(e, more * leaves, bc, bh, g)
        key, hit = _leaf_set(e, pts, lo)
        if key.numel() >= leaves:
            break
    if key.numel() > leaves:
        rank = torch.rand(key.numel(), device=DEV, generator=g) + hit.float()
        key = key[torch.argsort(rank, descending=True)[:leaves]]
    key = torch.sort(key).values
    n = key.numel()
    dens = torch.empty((n, 8), device=DEV)
    boxes = [(torch.tensor(c, dtype=torch.float32, device=DEV), torch.tensor(h, dtype=torch.float32, device=DEV))
             for c, h in zip(bc, bh)]
    m19 = (1 << 19) - 1
    for a in range(0, n, 2_000_000):
        k = key[a:a + 2_000_000]
        s = e.root * torch.exp2(-(k >> 57).float())
        mn = torch.stack([k & m19, (k >> 19) & m19, (k >> 38) & m19], 1) * s[:, None] + lo
        corner = mn[:, None, :] + off.float() * s[:, None, None]
        d = corner[..., 2].abs()
        for c, h in boxes:
            d = torch.minimum(d, _box_distance(corner, c, h))
        hi = (3.0 / s)[:, None] * torch.exp(0.25 * torch.randn(k.numel(), 8, device=DEV, generator=g))
        dens[a:a + 2_000_000] = V_FAR + (hi - V_FAR) * torch.exp(-2.0 * (d / s[:, None]).square())
    coef = 0.1 * torch.randn(n, (sh + 1) ** 2, 3, device=DEV, generator=g)
    return dv.DeviceOctree(key, dens, coef, sh, (0.0, 0.0, e.cz), e.root, dv.DV_ROLE_BG, max_level=e.lmax), pts


def _actor_cells(cells):
    """Grid cells of a 4.5 x 1.9 x 1.6 m body nearest to its surface, and their corners' distance to it."""
    dims = torch.tensor([4.5, 1.9, 1.6], dtype=torch.float64, device=DEV)
    root, clip, level = 1.2 * 4.5, 0.6 * dims, 6 if cells <= 30_000 else 7
    s = root / (1 << level)
    lo = torch.ceil((root / 2 - clip) / s - 1e-9).long().tolist()
    hi = torch.floor((root / 2 + clip) / s + 1e-9).long().tolist()
    ijk = torch.cartesian_prod(*[torch.arange(a, b, device=DEV) for a, b in zip(lo, hi)])
    body = dims / 2 * torch.tensor([0.95, 0.9, 0.9], dtype=torch.float64, device=DEV)
    zero = torch.zeros(3, dtype=torch.float64, device=DEV)
    order = torch.argsort(_box_distance(-root / 2 + (ijk + 0.5) * s, zero, body), stable=True)[:cells]
    ijk = ijk[torch.sort(order).values]
    corner = -root / 2 + (ijk[:, None, :] + torch.tensor(_OFF, device=DEV)) * s
    key = torch.sort(_pack(level, ijk[:, 0], ijk[:, 1], ijk[:, 2]))
    return key.values, _box_distance(corner, zero, body)[key.indices].float(), s, root, level, tuple(clip.tolist())


def _actors(n, cells, sh, seed):
    if n == 0:
        return []
    key, dist, s, root, level, clip = _actor_cells(cells)
    g, fall, out = _gen(seed + 2000), torch.exp(-2.0 * (dist / s).square()), []
    for _ in range(n):
        hi = (3.0 / s) * torch.exp(0.25 * torch.randn(dist.shape, device=DEV, generator=g))
        coef = 0.1 * torch.randn(key.numel(), (sh + 1) ** 2, 3, device=DEV, generator=g)
        out.append(dv.DeviceOctree(key, V_FAR + (hi - V_FAR) * fall, coef, sh, (0.0, 0.0, 0.0), root,
                                   dv.DV_ROLE_ACTOR, clip, level))
    return out


def _lanes(n, seed):
    """Straight lanes: a start point per actor (boxes disjoint where there is room), a heading, a speed."""
    rng, out = random.Random(seed + 1000), []
    x1 = 8.0 + 6.0 * max(n, 6) if n > 8 else 45.0
    tries = 0
    while len(out) < n:
        tries += 1
        p = (rng.uniform(8.0, x1), rng.uniform(-9.0, 9.0))
        if tries < 20000 and any(math.hypot(p[0] - q[0][0], p[1] - q[0][1]) < 6.9 for q in out):
            continue
        out.append((p, rng.uniform(-math.pi, math.pi), rng.uniform(5.0, 15.0)))
    return out


def _poses(lanes, t):
    return [_identity()] + [_pose(_rot_z(a), (p[0] + v * t * math.cos(a), p[1] + v * t * math.sin(a), 0.8)) for p, a, v in lanes]


def _street(case, seed):
    bg, cloud = _background(case["leaves"], case["sh"], seed)
    return [bg] + _actors(case["actors"], case["cells"], case["sh"], seed), _lanes(case["actors"], seed), cloud


def _surround(case, seed):
    """The call's cameras around the vehicle; the first looks along the road."""
    rng = random.Random(seed + 77)
    pos, n = (rng.uniform(-0.5, 0.5), rng.uniform(-0.5, 0.5), 1.8), case["cams"]
    far = 800.0 if case.get("leaves", 0) > 12_000_000 else 400.0
    return [_vehicle_camera(case["W"], case["H"], rng.uniform(-0.02, 0.02) + 2 * math.pi * c / max(n, 6), pos, far)
            for c in range(n)]


def _upstream(n_pix, g, normals):
    u = [torch.randn(n_pix, 3, device=DEV, generator=g), 0.01 * torch.randn(n_pix, device=DEV, generator=g),
         torch.randn(n_pix, device=DEV, generator=g)]
    return u + [torch.randn(n_pix, 3, device=DEV, generator=g)] if normals else u


def _grid_scene(case, seed):
    g, n = _gen(seed), 1 << case["level"]
    ax = torch.arange(n, device=DEV)
    ijk = torch.cartesian_prod(ax, ax, ax)
    V = ijk.shape[0]
    dens = torch.exp(torch.randn(V, 8, device=DEV, generator=g))
    sh = (torch.rand(V, 1, 3, device=DEV, generator=g) - 0.5) / SH_C0
    key = _pack(case["level"], ijk[:, 2], ijk[:, 1], ijk[:, 0])
    oc = dv.DeviceOctree(key, dens, sh, 0, (0.0, 0.0, 0.0), 2.0, dv.DV_ROLE_BG, max_level=case["level"])
    rng = random.Random(seed)
    az, el = math.radians(30.0 + rng.uniform(-10, 10)), math.radians(20.0 + rng.uniform(-5, 5))
    eye = 2.5 * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
    cam = _camera(case["W"], case["H"], _look(eye, (0.0, 0.0, 0.0)), 0.1, 100.0)
    return oc, cam, _upstream(case["W"] * case["H"], g, False)


def _slots(case, seed):
    """Slot lists with a render's structure: a pixel meets ``slots`` voxels front to back on average, a voxel
    covers a rectangle of a few to a few tens of pixels, and the weights are those of alpha compositing."""
    g = _gen(seed)
    W, H, m = case["W"], case["H"], case["slots"]
    y, x = torch.meshgrid(torch.arange(H, device=DEV), torch.arange(W, device=DEV), indexing="ij")
    x, y = x.reshape(-1), y.reshape(-1)
    vox, first, layers = [], 0, 2 * m
    for k in range(layers):
        c, ox, oy = 6 + (7 * k) % 35, (11 * k) % 41, (17 * k) % 41
        nx, ny = (W + ox) // c + 1, (H + oy) // c + 1
        vox.append(first + (y + oy) // c * nx + (x + ox) // c)
        first += nx * ny
    vox = torch.stack(vox, 1)
    # half of the layers' voxels do not exist (empty space)
    alive = (torch.rand(first, device=DEV, generator=g) < 0.5)[vox]
    tau = (torch.exp(torch.randn(first, device=DEV, generator=g) - 2.5))[vox] * alive
    T = torch.exp(-torch.cumsum(tau, 1))
    w = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1) - T
    off = torch.zeros(W * H + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(alive.sum(1), 0)
    return off, vox[alive].int(), w[alive].contiguous(), first, g


RESOLUTIONS = ((480, 270), (960, 540), (1920, 1080))


# ---------------------------------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------------------------------

def prepare(case, seed):
    s = SimpleNamespace(case=case, opts=dv.make_opts(K=case.get("K", 1)))
    kind = case["kind"]
    if kind == "grid_train":
        oc, cam, s.up = _grid_scene(case, seed)
        s.octs, s.poses, s.cams = [oc], [_identity()], [cam]
        s.dens, s.sh = [oc.dens.requires_grad_()], [oc.sh.requires_grad_()]
        return s
    if kind == "features":
        off, vox, w, n_vox, g = _slots(case, seed)
        s.weights, C = dv.Weights(off, vox, w), case["channels"]
        s.feat = torch.randn(n_vox, C, device=DEV, generator=g)
        s.feat2d = torch.randn(case["W"] * case["H"], C, device=DEV, generator=g)
        s.accum, s.wsum = torch.empty_like(s.feat), torch.empty(n_vox, device=DEV)
        return s
    if kind == "sky":
        g = _gen(seed)
        s.cams = _surround(case, seed)
        n = case["W"] * case["H"] * case["cams"]
        s.env = torch.rand(case["He"], case["We"], 3, device=DEV, generator=g)
        # a street's alpha: nearly opaque ground and buildings, clear sky above the horizon
        row = (torch.arange(n, device=DEV) // case["W"]) % case["H"]
        sky = (row < 0.55 * case["H"]) & (torch.rand(n, device=DEV, generator=g) < 0.8)
        s.alpha = torch.where(sky, 0.05, 0.97) * torch.rand(n, device=DEV, generator=g).sqrt()
        s.rgb = torch.rand(n, 3, device=DEV, generator=g) * s.alpha[:, None]
        s.d_out = torch.randn(n, 3, device=DEV, generator=g)
        s.d_env, s.d_alpha = torch.empty_like(s.env), torch.empty_like(s.alpha)
        return s
    if kind == "init":
        bg, s.cloud = _background(case["leaves"], 0, seed)
        s.key, s.center, s.root, s.level = bg.key, bg.center, bg.root_size, bg.max_level
        s.cloud = s.cloud.contiguous()
        s.cams = _surround(case, seed)
        return s
    s.octs, lanes, _ = _street(case, seed)
    if kind == "serve":
        rng = random.Random(seed + 5)
        sizes = [RESOLUTIONS[r % 3] for r in range(case["requests"])]
        n = [W * H for W, H in sizes]
        s.images = (torch.empty(sum(n), 3, device=DEV), torch.empty(sum(n), device=DEV), torch.empty(sum(n), device=DEV))
        outs = zip(*(t.split(n) for t in s.images))
        s.requests = [(_vehicle_camera(W, H, 0.0, (-50.0 + 100.0 * rng.random(), 0.0, 1.8)),
                       _poses(lanes, 10.0 * rng.random()), out) for (W, H), out in zip(sizes, outs)]
        s.server = dv.Server(s.octs, max_views=case["max_views"], n_workers=case["workers"], opts=s.opts)
        return s
    s.cams, s.poses = _surround(case, seed), _poses(lanes, 0.0)
    n_pix = case["W"] * case["H"] * case["cams"]
    if kind == "lift":
        g, C = _gen(seed + 3), case["channels"]
        rgb, depth, alpha, s.state = dv.dv_render(s.octs, s.poses, s.cams, s.opts, save_state=True)
        n_vox = sum(o.n for o in s.octs)
        s.feat = torch.randn(n_vox, C, device=DEV, generator=g)
        s.feat2d = torch.randn(n_pix, C, device=DEV, generator=g)
        s.accum, s.wsum = torch.empty_like(s.feat), torch.empty(n_vox, device=DEV)
        return s
    if kind == "train":
        s.up = _upstream(n_pix, _gen(seed + 3), case["normals"])
        if case["shared"]:
            # the background's densities live on shared grid corners (one per distinct point, in buffers
            # with room for the most a leaf set of this size can have)
            bg = s.octs[0]
            grid, s.index = dv.dv_shared_corners(bg.key, bg.max_level)
            s.index = s.index.contiguous()
            s.corner = torch.full((8 * bg.n,), V_FAR, device=DEV)
            s.corner.scatter_reduce_(0, s.index.long().reshape(-1), bg.dens.reshape(-1), "amax")
            s.d_corner = torch.empty_like(s.corner)
        s.dens, s.sh = [o.dens for o in s.octs], [o.sh for o in s.octs]
        s.autograd = case["cams"] == 1 and not case["shared"]
        if s.autograd:
            s.dens, s.sh = [t.requires_grad_() for t in s.dens], [t.requires_grad_() for t in s.sh]
            return s
        # one flat gradient buffer for all octrees' densities and one for their coefficients
        nd, ns = [o.dens.numel() for o in s.octs], [o.sh.numel() for o in s.octs]
        s.g_dens, s.g_sh = torch.empty(sum(nd), device=DEV), torch.empty(sum(ns), device=DEV)
        s.v_dens = [v.view_as(o.dens) for v, o in zip(s.g_dens.split(nd), s.octs)]
        s.v_sh = [v.view_as(o.sh) for v, o in zip(s.g_sh.split(ns), s.octs)]
    return s


def _padded(t, n):
    return torch.nn.functional.pad(t, (0, n - t.numel()))


def _autograd_step(s, normals=False):
    out = dv.render(s.octs, s.poses, s.cams, s.opts, dens=s.dens, sh=s.sh, normals=normals)
    grads = torch.autograd.grad(out, s.dens + s.sh, s.up)
    return {"images": [t.detach() for t in out], "grads": list(grads)}


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "grid_train":
        return _autograd_step(s)
    if kind == "render":
        return dv.dv_render(s.octs, s.poses, s.cams, s.opts)[:3]
    if kind == "train":
        if s.autograd:
            return _autograd_step(s, case["normals"])
        # the same step through the ABI-named calls, accumulating into the program's own buffers
        dens = None
        if case["shared"]:
            dens = [dv.dv_corner_gather(s.index, s.corner)] + s.dens[1:]
        out = dv.dv_render(s.octs, s.poses, s.cams, s.opts, save_state=True, dens=dens,
                           sh=None if dens is None else s.sh, normals=case["normals"])
        s.g_dens.zero_()
        s.g_sh.zero_()
        up = s.up
        dv.dv_render_backward(out[-1], up[0], up[1], up[2], s.v_dens, s.v_sh, d_normal=up[3] if case["normals"] else None)
        dv.dv_state_free(out[-1])
        res = {"images": list(out[:-1]), "g_dens": s.g_dens, "g_sh": s.g_sh}
        if case["shared"]:
            s.d_corner.zero_()
            dv.dv_corner_scatter(s.index, s.v_dens[0], s.d_corner)
            res["d_corner"] = s.d_corner
        return res
    if kind in ("lift", "features"):
        w = dv.dv_state_weights(s.state) if kind == "lift" else s.weights
        F = dv.dv_features_render(w, s.feat)
        s.accum.zero_()
        s.wsum.zero_()
        dv.dv_features_fuse(w, s.feat2d, s.accum, s.wsum)
        return {"features": F, "accum": s.accum, "wsum": s.wsum}
    if kind == "init":
        step = s.root / (1 << s.level)
        kept = dv.dv_visibility_prune(s.key, s.level, s.center, s.root, s.cams, 0.0)
        grid, index = dv.dv_shared_corners(s.key, s.level)
        corner = dv.dv_soft_prior(grid, s.center, s.root, s.level, s.cloud, step, V_CLOSE, V_FAR)
        dens = dv.dv_corner_gather(index, corner)
        finer = dv.dv_subdivide_round(s.key, s.level, s.center, s.root, s.cloud, step)
        # the program's own arrays have room for the most a call can return
        room = 8 * s.key.numel()
        return {"kept": _padded(kept, room), "grid": _padded(grid, room), "index": index, "corner": _padded(corner, room),
                "dens": dens, "finer": _padded(finer, room)}
    if kind == "sky":
        out = dv.dv_sky_composite(s.cams, s.env, s.rgb, s.alpha)
        s.d_env.zero_()
        s.d_alpha.zero_()
        dv.dv_sky_backward(s.cams, s.env, s.alpha, s.d_out, s.d_env, s.d_alpha)
        return {"rgb": out, "d_env": s.d_env, "d_alpha": s.d_alpha}
    # serve: the requests queue up while admission is held, then run in the batches the server forms
    s.server.pause(True)
    tickets = [s.server.submit(cam, poses, out) for cam, poses, out in s.requests]
    s.server.pause(False)
    for t in tickets:
        s.server.wait(t)
        s.server.release(t)
    return s.images


# ---------------------------------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "sky":
        n, m = case["W"] * case["H"] * case["cams"], case["He"] * case["We"] * 12
        # forward: rgb, alpha in, rgb out; backward: upstream and alpha in, d_alpha out; the map in, its gradient out
        return {"bytes": n * (28 + 20) + 2 * m, "flops": n * 120}
    if kind == "init":
        n = case["leaves"]
        pts = 2.5 * n
        # keys in (three calls read the same ones), corner indices and densities out, points in, new keys out
        return {"bytes": 8 * n + 32 * n + 32 * n + 16 * n + 12 * pts + 16 * n, "flops": 400 * n + 100 * pts}
    if kind == "features":
        n, C = case["W"] * case["H"], case["channels"]
        slots, vox = n * case["slots"], n * case["slots"] // 300
        return {"bytes": 8 * slots + 8 * n + 8 * n * C + 8 * vox * C, "flops": 4 * slots * C}
    if kind == "grid_train":
        n, V = case["W"] * case["H"], 8 ** case["level"]
        return {"bytes": n * 40 + V * (8 + 2 * (32 + 12)), "flops": n * 11 * (40 + 47 + 66 + 59 * case["K"])}
    if kind == "serve":
        n = sum(RESOLUTIONS[r % 3][0] * RESOLUTIONS[r % 3][1] for r in range(case["requests"]))
        cams = case["requests"]
    else:
        n, cams = case["W"] * case["H"] * case["cams"], case["cams"]
    V, row = case["leaves"] + case["actors"] * case["cells"], 32 + 12 * (case["sh"] + 1) ** 2
    seen = min(1.0, 0.2 * min(cams, 6)) * V  # a 60 degree camera sees about a fifth of the leaves
    segs = 17 * n
    if kind == "lift":
        C = case["channels"]
        return {"bytes": 8 * segs + 8 * n + 8 * n * C + 8 * seen * C, "flops": segs * (60 + 47 + 4 * C)}
    b = 8 * V + row * seen + 20 * n
    f = segs * (60 + 16 + 31 * case.get("K", 1))
    if kind == "train":
        N = 12 if case["normals"] else 0
        b += n * (20 + 2 * N) + row * V  # upstream gradients in, every gradient row out
        f += segs * (60 + 59 + 66 * case["K"])
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------------------------
# 64-bit values of what can be computed in a few seconds without the renderer
# ---------------------------------------------------------------------------------------------------

def _cam_dirs(cam):
    """Unit ray directions in world axes [P, 3], row-major over the image, and the camera centre."""
    u = torch.arange(cam.W, dtype=torch.float64, device=DEV) + 0.5
    v = torch.arange(cam.H, dtype=torch.float64, device=DEV) + 0.5
    f32 = lambda a: float(np.float32(a))
    y, x = torch.meshgrid((v - f32(cam.cy)) / f32(cam.fy), (u - f32(cam.cx)) / f32(cam.fx), indexing="ij")
    d = torch.stack([x, y, torch.ones_like(x)], -1).reshape(-1, 3)
    d = d / d.norm(dim=1, keepdim=True)
    R = torch.tensor(cam.pose.R.astype(np.float64), device=DEV)
    return d @ R.T, torch.tensor(cam.pose.t.astype(np.float64), device=DEV)


def _exact_grid(case, seed):
    """The plain per-ray definition in 64 bits: every ray against every voxel, sorted by entry, composited."""
    oc, cam, up = _grid_scene(case, seed)
    n, K, eps = 1 << case["level"], case["K"], float(np.float32(1e-4))
    s = 2.0 / n
    m19 = (1 << 19) - 1
    mn = torch.stack([oc.key & m19, (oc.key >> 19) & m19, (oc.key >> 38) & m19], 1).double() * s - 1.0
    dens, sh = oc.dens.double().requires_grad_(), oc.sh.double().requires_grad_()
    dirs, o = _cam_dirs(cam)
    near, far = float(np.float32(cam.near)), float(np.float32(cam.far))
    images = []
    g_dens, g_sh = torch.zeros_like(dens), torch.zeros_like(sh)
    step = max(1, 30_000_000 // mn.shape[0])
    for a in range(0, dirs.shape[0], step):
        d, color = dirs[a:a + step], (SH_C0 * sh[:, 0, :] + 0.5).clamp(min=0.0)
        lo = torch.full((d.shape[0], mn.shape[0]), near, dtype=torch.float64, device=DEV)
        hi = torch.full_like(lo, far)
        for k in range(3):
            dk = d[:, k:k + 1]
            dk = torch.where(dk.abs() < 1e-20, torch.full_like(dk, 1e-20), dk)
            ta, tb = (mn[:, k] - o[k]) / dk, (mn[:, k] + s - o[k]) / dk
            lo, hi = torch.maximum(lo, torch.minimum(ta, tb)), torch.minimum(hi, torch.maximum(ta, tb))
        lo = torch.where(hi > lo, lo, torch.full_like(lo, math.inf))
        t0, idx = torch.topk(lo, min(3 * n + 2, mn.shape[0]), dim=1, largest=False)
        t1 = torch.gather(hi, 1, idx)
        hit = torch.isfinite(t0)
        t0, t1 = torch.where(hit, t0, 0.0), torch.where(hit, t1, 0.0)
        sig = torch.zeros_like(t0)
        rho, base = dens[idx], mn[idx]
        for q in range(K):
            t = t0 + (t1 - t0) * (q + 0.5) / K
            p = ((o + t[..., None] * d[:, None, :] - base) / s).clamp(0.0, 1.0)
            w = torch.stack([(p[..., 0] if c & 1 else 1 - p[..., 0]) * (p[..., 1] if c & 2 else 1 - p[..., 1]) *
                             (p[..., 2] if c & 4 else 1 - p[..., 2]) for c in range(8)], -1)
            r = (w * rho).sum(-1)
            sig = sig + torch.where(r > 1.1, r, 1.1 * torch.exp(r.clamp(max=1.1) / 1.1 - 1.0))
        tau = torch.where(hit, (t1 - t0) / K * sig, 0.0)
        T_end = torch.exp(-torch.cumsum(tau, 1))
        T = torch.cat([torch.ones_like(T_end[:, :1]), T_end[:, :-1]], 1)
        live = T.detach() >= eps  # the first segment that brings T below eps is the last one
        wgt = torch.where(live, T - T_end, 0.0)
        out = [(wgt[..., None] * color[idx]).sum(1), (wgt * 0.5 * (t0 + t1)).sum(1), wgt.sum(1)]
        gd, gs = torch.autograd.grad(out, [dens, sh], [u[a:a + step].double() for u in up])
        g_dens += gd
        g_sh += gs
        images.append([t.detach() for t in out])
    return {"images": [torch.cat(x) for x in zip(*images)], "grads": [g_dens, g_sh]}


def _exact_sky(s):
    He, We = s.env.shape[:2]
    env, off = s.env.double().reshape(-1, 3), 0
    out, d_alpha, d_env = [], [], torch.zeros_like(env)
    for cam in s.cams:
        d, _ = _cam_dirs(cam)
        n = d.shape[0]
        x = (torch.atan2(d[:, 1], d[:, 0]) + math.pi) * (We / (2 * math.pi)) - 0.5
        y = torch.acos(d[:, 2].clamp(-1, 1)) * (He / math.pi) - 0.5
        x0, y0 = x.floor(), y.floor()
        fx, fy = x - x0, y - y0
        T = 1.0 - s.alpha[off:off + n].double()
        g = s.d_out[off:off + n].double()
        sky = torch.zeros_like(g)
        for a, b, w in ((0, 0, (1 - fx) * (1 - fy)), (1, 0, fx * (1 - fy)), (0, 1, (1 - fx) * fy), (1, 1, fx * fy)):
            t = (y0 + b).clamp(0, He - 1).long() * We + ((x0 + a).long() % We)
            sky += w[:, None] * env[t]
            d_env.index_add_(0, t, (T * w)[:, None] * g)
        out.append(s.rgb[off:off + n].double() + T[:, None] * sky)
        d_alpha.append(-(g * sky).sum(1))
        off += n
    return {"rgb": torch.cat(out), "d_env": d_env.view(s.env.shape), "d_alpha": torch.cat(d_alpha)}


def _exact_features(s):
    w, P = s.weights, s.feat2d.shape[0]
    pix = torch.repeat_interleave(torch.arange(P, device=DEV), w.offsets[1:] - w.offsets[:-1])
    vox, wt = w.voxel.long(), w.weight.double()
    n_vox, C = s.feat.shape
    F = torch.empty(P, C, dtype=torch.float64, device=DEV)
    acc = torch.empty(n_vox, C, dtype=torch.float64, device=DEV)
    for c in range(0, C, 16):
        f, f2 = s.feat[:, c:c + 16].double(), s.feat2d[:, c:c + 16].double()
        F[:, c:c + 16] = torch.zeros(P, f.shape[1], dtype=torch.float64, device=DEV).index_add_(0, pix, wt[:, None] * f[vox])
        acc[:, c:c + 16] = torch.zeros(n_vox, f.shape[1], dtype=torch.float64, device=DEV).index_add_(0, vox, wt[:, None] * f2[pix])
    ws = torch.zeros(n_vox, dtype=torch.float64, device=DEV).index_add_(0, vox, wt)
    return {"features": F, "accum": acc, "wsum": ws}


def _exact_prior(s):
    """Densities of the distinct corners of the leaves from the nearest point, in 64 bits.  Points farther than
    three steps change a density by less than 1e-7 (far below a 32-bit rounding of it) and are left out."""
    m19, L = (1 << 19) - 1, s.level
    lv = s.key >> 57
    ijk = torch.stack([s.key & m19, (s.key >> 19) & m19, (s.key >> 38) & m19], 1)
    c = (ijk[:, None, :] + torch.tensor(_OFF, device=DEV)) << (L - lv)[:, None, None]
    grid, index = torch.unique((c[..., 2] << 42) | (c[..., 1] << 21) | c[..., 0], return_inverse=True)
    m21, step = (1 << 21) - 1, s.root / (1 << L)
    q = torch.stack([grid & m21, (grid >> 21) & m21, (grid >> 42) & m21], 1).double() * step
    lo = torch.tensor(s.center, dtype=torch.float64, device=DEV) - 0.5 * s.root
    p = s.cloud.double() - lo
    h = 3.0 * float(np.float32(step)) * (1 + 1e-9)
    cell = lambda v: torch.floor(v / h).long() + (1 << 19)
    code = lambda v: (v[:, 2] << 42) | (v[:, 1] << 21) | v[:, 0]
    key, order = torch.sort(code(cell(p)))
    p, qc = p[order], cell(q)
    best = torch.full((q.shape[0],), math.inf, dtype=torch.float64, device=DEV)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            a = torch.searchsorted(key, code(qc + torch.tensor([-1, dy, dz], device=DEV)))
            n = torch.searchsorted(key, code(qc + torch.tensor([1, dy, dz], device=DEV)), right=True) - a
            ends = torch.cumsum(n, 0)
            at = 0
            while at < q.shape[0]:
                base = int(ends[at - 1]) if at else 0
                to = max(at + 1, int(torch.searchsorted(ends, torch.tensor(base + 50_000_000, device=DEV), right=True)))
                cnt = n[at:to]
                who = torch.repeat_interleave(torch.arange(at, min(to, q.shape[0]), device=DEV), cnt)
                pos = torch.arange(who.numel(), device=DEV) - (ends[who] - n[who] - base) + a[who]
                best.scatter_reduce_(0, who, (p[pos] - q[who]).square().sum(1), "amin")
                at = to
    sm = float(np.float32(step))
    corner = V_FAR + (V_CLOSE - V_FAR) * torch.exp(-2.0 * best / (sm * sm))
    return _padded(corner, 8 * s.key.numel()), corner[index.reshape(-1, 8)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "grid_train":
        return _exact_grid(case, seed)
    if kind == "sky":
        return _exact_sky(prepare(case, seed))
    if kind == "features":
        return _exact_features(prepare(case, seed))
    if kind == "init":
        corner, dens = _exact_prior(prepare(case, seed))
        return {"kept": None, "grid": None, "index": None, "corner": corner, "dens": dens, "finer": None}
    return None
