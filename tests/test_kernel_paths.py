"""Sizes at which the kernels change their way of working: crowded actor tiles (a CTA per pixel block) and rays
through more actor boxes than a ray has slots, voxels from many pixels down to less than one (lists per lane or
lockstep in the backward), the projection's queue, the counted sort, the initialisation's FP32 decisions (ties,
clouds far from the origin, thresholds far below and above a leaf), and sky lookups that share a cell.

References: the FP64 oracle and the tolerances of helpers.py; whole numbers and flags bit for bit.  The soft prior
is float32 of an FP64 value of at most 10 (1e-5 absolute, as in the parity tests of the initialisation)."""
import numpy as np
import pytest

import oracle
import oracle.init as oi
import oracle.sky as osky
import synth
from helpers import check_forward, check_grads, device_scene, gpu_render, orbit, split_images

N_ATOL = 1e-4  # normals, as in their parity tests


def _grid(level, frac, rng, n=None):
    m = 1 << level
    c = np.flatnonzero(rng.uniform(size=m ** 3) < frac) if n is None else np.sort(rng.choice(m ** 3, n, replace=False))
    return synth.pack_keys(np.full(c.size, level), c % m, (c // m) % m, c // (m * m))


def _octree(key, scale, rng, root, role=synth.BG, half=None, degree=1):
    V = key.size
    dens = (rng.lognormal(0.0, 0.8, (V, 8)) * scale).astype(np.float32)
    sh = rng.normal(0, 0.3, (V, (degree + 1) ** 2, 3)).astype(np.float32)
    args = () if half is None else (half,)
    return synth.Octree(key, dens, sh, degree, (0.0, 0.0, 0.0), root, role, *args)


def _row_of_actors(n, level):
    """n thin actors one behind the other on the camera's axis, each turned about it: the ray through the
    image's middle has n intervals.  Returns the scene, the camera and the most crowded tile's voxel centres."""
    rng = np.random.default_rng(100 * n + level)
    root, half, gap = 0.7, (0.08, 0.3, 0.3), 0.25
    octs = [_octree(_grid(3, 0.4, rng), 0.02, rng, 4.0)]
    poses = [synth.Pose()]
    cam = synth.pinhole(40, 34, 12.0, synth.look_at((-6.0, 0.0, 0.0), (0.0, 0.0, 0.0)), 0.1, 60.0)
    count = np.zeros((3, 3), np.int64)
    for a in range(n):
        o = _octree(_grid(level, 0.6, rng), 1.5 / n, rng, root, synth.ACTOR, half)
        w = rng.uniform(0, 2 * np.pi)
        R = np.array([[1, 0, 0], [0, np.cos(w), -np.sin(w)], [0, np.sin(w), np.cos(w)]])
        pose = synth.Pose(R, np.array([gap * a, 0.0, 0.0]))
        octs.append(o)
        poses.append(pose)
        _, i, j, k = oi._unpack(o.key)
        c = (np.stack([i, j, k], 1) + 0.5) * (root / 2 ** level) - 0.5 * root
        c = c[(np.abs(c) < half).all(1)] @ R.T + pose.t
        pc = (c - np.asarray(cam.pose.t)) @ np.asarray(cam.pose.R).reshape(3, 3)
        u = (cam.fx * pc[:, 0] / pc[:, 2] + cam.cx).astype(int) // 16
        v = (cam.fy * pc[:, 1] / pc[:, 2] + cam.cy).astype(int) // 16
        np.add.at(count, (v, u), 1)
    return synth.Scene(octs, poses), cam, count.max()


# 1 to 4 and 5 or more boxes on a tile; up to 8, 9 to 32 and more than 32 intervals on a ray; few and many pairs; the
# code for one sample and for several
@pytest.mark.gpu
@pytest.mark.parametrize("K", [2, 1])
@pytest.mark.parametrize("n,level,crowded", [(3, 5, True), (7, 4, True), (14, 4, True), (36, 4, True), (12, 1, False)])
def test_actor_tiles(dv, n, level, crowded, K):
    import torch
    sc, cam, most = _row_of_actors(n, level)
    assert most >= 1023 if crowded else most < 300
    P = cam.W * cam.H
    rng = np.random.default_rng(n)
    g = [np.float64(np.float32(x)) for x in (rng.normal(size=(P, 3)), 0.1 * rng.normal(size=P), rng.normal(size=P),
                                             rng.normal(size=(P, 3)))]
    ds = device_scene(sc)
    opts = dv.make_opts(K, 1e-4)
    rgb, depth, alpha, nrm, st = dv.dv_render(ds, sc.poses, [cam], opts, save_state=True, normals=True)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")
    d_dens = [torch.zeros_like(o.dens) for o in ds]
    d_sh = [torch.zeros_like(o.sh) for o in ds]
    dv.dv_render_backward(st, t(g[0]), t(g[1]), t(g[2]), d_dens, d_sh, d_normal=t(g[3]))
    torch.cuda.synchronize()
    st.free()
    o = oracle.render(sc.octrees, sc.poses, cam, oracle.Opts(K, 1e-4), normals=True)
    im = lambda x, c=None: split_images(x.cpu().numpy(), [cam], c)[0]
    check_forward(im(rgb, 3), im(depth), im(alpha), o[0], o[1], o[2], f"{n} actors")
    assert np.abs(im(nrm, 3) - o[4]).max() <= N_ATOL
    od, os_ = oracle.backward(sc.octrees, sc.poses, cam, g[0], g[1], g[2], oracle.Opts(K, 1e-4), g_normal=g[3])
    check_grads([x.cpu().numpy() for x in d_dens], od, f"{n} actors d_dens")
    check_grads([x.cpu().numpy() for x in d_sh], os_, f"{n} actors d_sh")
    # the exported weights of a pixel add up to its alpha
    rgb, depth, alpha, st = dv.dv_render(ds, sc.poses, [cam], opts, save_state=True)
    W = dv.dv_state_weights(st)
    off = W.offsets.cpu().numpy()
    w = W.weight.cpu().numpy().astype(np.float64)
    st.free()
    total = np.add.reduceat(np.append(w, 0.0), np.minimum(off[:-1], w.size)) * (np.diff(off) > 0)
    assert np.abs(total - alpha.cpu().numpy().ravel()).max() <= 1e-5


# rays that reach an actor whose partial composite was left out or stopped early, both of which assume T <= 1:
# behind negative densities under the identity activation (T of some 5 in front of the actors), and with eps_stop
# above 1 (a ray then ends with its first segment).  Values follow T, so the bounds are relative to the largest
@pytest.mark.gpu
@pytest.mark.parametrize("n,level", [(3, 5), (7, 4), (12, 1)])
@pytest.mark.parametrize("eps,identity", [(0.3, True), (2.0, False)])
def test_actor_partials_behind_transmittance_above_one(dv, n, level, eps, identity):
    import torch
    sc, cam, _ = _row_of_actors(n, level)
    if identity:
        sc.octrees[0].dens *= np.float32(-40.0)
        for o in sc.octrees[1:]:
            o.dens *= np.float32(9.0 * n)
    act = oracle.ACT_IDENTITY if identity else oracle.ACT_EXPLIN
    P = cam.W * cam.H
    rng = np.random.default_rng(n)
    g = [np.float64(np.float32(x)) for x in (rng.normal(size=(P, 3)), 0.1 * rng.normal(size=P), rng.normal(size=P))]
    ds = device_scene(sc)
    rgb, depth, alpha, st = dv.dv_render(ds, sc.poses, [cam], dv.make_opts(1, eps, act), save_state=True)
    W = dv.dv_state_weights(st)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")
    d_dens = [torch.zeros_like(o.dens) for o in ds]
    d_sh = [torch.zeros_like(o.sh) for o in ds]
    dv.dv_render_backward(st, t(g[0]), t(g[1]), t(g[2]), d_dens, d_sh)
    torch.cuda.synchronize()
    st.free()
    o = oracle.render(sc.octrees, sc.poses, cam, oracle.Opts(1, eps, act))
    for x, ref, tol in ((rgb, o[0], 1e-4), (depth, o[1], 1e-3), (alpha, o[2], 1e-4)):
        assert np.abs(x.cpu().numpy().reshape(ref.shape) - ref).max() <= tol * np.abs(ref).max()
    off, w = W.offsets.cpu().numpy(), W.weight.cpu().numpy().astype(np.float64)
    total = np.add.reduceat(np.append(w, 0.0), np.minimum(off[:-1], w.size)) * (np.diff(off) > 0)
    assert np.abs(total - alpha.cpu().numpy().ravel()).max() <= 1e-4 * max(1.0, np.abs(o[2]).max())
    od, os_ = oracle.backward(sc.octrees, sc.poses, cam, g[0], g[1], g[2], oracle.Opts(1, eps, act))
    check_grads([x.cpu().numpy() for x in d_dens], od, f"{n} actors d_dens")
    check_grads([x.cpu().numpy() for x in d_sh], os_, f"{n} actors d_sh")


# every exported slot is written, also where the transmittance behind an actor is within rounding of eps_stop: an
# interval's replay from its entry may then stop before segments that the forward, applying its partial, counted.
# The actor is a dense slab and a long tail of segments without weight; eps_stop goes through the floats around a
# pixel's final transmittance
@pytest.mark.gpu
def test_export_writes_every_slot(dv):
    import torch
    rng = np.random.default_rng(4)
    key = _grid(2, 0.0, rng, 64)
    bg = _octree(key[oi._unpack(key)[1] < 2], 0.05, rng, 4.0)  # nothing behind the actor's slab
    actor = _octree(_grid(4, 0.0, rng, 4096), 1.0, rng, 0.8, synth.ACTOR, (0.4, 0.4, 0.4))
    actor.dens[oi._unpack(actor.key)[1] >= 6] = -60.0
    sc = synth.Scene([bg, actor], [synth.Pose(), synth.Pose()])
    cam = synth.pinhole(16, 8, 6.0, synth.look_at((-6.0, 0.0, 0.0), (0.0, 0.0, 0.0)), 0.1, 60.0)
    ds = device_scene(sc)
    T = 1.0 - dv.dv_render(ds, sc.poses, [cam], dv.make_opts(1, 0.0))[2].cpu().numpy().astype(np.float64)
    assert T.min() > 0.25 and T.max() < 0.5
    for p in range(0, cam.W * cam.H, 2):
        for j in range(-4, 5):
            eps = float(np.float32(T[p] + j * 2.0 ** -25))
            alpha, st = dv.dv_render(ds, sc.poses, [cam], dv.make_opts(1, eps), save_state=True)[2:]
            W = dv.dv_state_weights(st)
            W.voxel.fill_(0x7fffffff)
            W.weight.fill_(float("nan"))
            dv.dv_state_weights(st, out=W)
            st.free()
            assert int(W.voxel.max()) < bg.n + actor.n and int(W.voxel.min()) >= 0
            pix = torch.repeat_interleave(torch.arange(cam.W * cam.H, device="cuda"), W.offsets.diff())
            total = torch.zeros(cam.W * cam.H, device="cuda").index_add_(0, pix, W.weight)
            assert float((total - alpha).abs().max()) <= 1e-5


# voxels of about 20, 5 and 0.6 pixels
@pytest.mark.gpu
@pytest.mark.parametrize("level,normals", [(1, False), (1, True), (3, True), (6, False), (6, True)])
def test_plain_backward_by_voxel_size(dv, level, normals):
    import torch
    rng = np.random.default_rng(level)
    sc = synth.Scene([_octree(_grid(level, 0.5 if level < 6 else 0.05, rng), 1.0, rng, 2.0)], [synth.Pose()])
    cam = orbit(33, 17, 40.0, 20.0)
    P = cam.W * cam.H
    g = [np.float64(np.float32(x)) for x in (rng.normal(size=(P, 3)), 0.1 * rng.normal(size=P), rng.normal(size=P),
                                             rng.normal(size=(P, 3)))]
    ds = device_scene(sc)
    out = dv.dv_render(ds, sc.poses, [cam], dv.make_opts(1, 1e-4), save_state=True, normals=normals)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")
    d_dens, d_sh = [torch.zeros_like(ds[0].dens)], [torch.zeros_like(ds[0].sh)]
    extra = {"d_normal": t(g[3])} if normals else {}
    dv.dv_render_backward(out[-1], t(g[0]), t(g[1]), t(g[2]), d_dens, d_sh, **extra)
    torch.cuda.synchronize()
    out[-1].free()
    extra = {"g_normal": g[3]} if normals else {}
    od, os_ = oracle.backward(sc.octrees, sc.poses, cam, g[0], g[1], g[2], oracle.Opts(1, 1e-4), **extra)
    check_grads([d_dens[0].cpu().numpy()], od, f"level {level} d_dens")
    check_grads([d_sh[0].cpu().numpy()], os_, f"level {level} d_sh")


# one voxel below the projection's queue, its first size, and a remainder; most voxels lie outside the frustum
@pytest.mark.gpu
@pytest.mark.parametrize("n", [99999, 131149, 399999, 400000, 431149])
def test_projection_queue(dv, n):
    rng = np.random.default_rng(n)
    sc = synth.Scene([_octree(_grid(6 if n < 64 ** 3 else 7, 0.0, rng, n), 0.5, rng, 8.0)], [synth.Pose()])
    cam = synth.pinhole(33, 21, 50.0, synth.look_at((0.3, -0.2, 0.1), (3.0, 1.0, 0.5)), 0.05, 3.0)
    rgb, depth, alpha, _ = gpu_render(device_scene(sc), sc.poses, [cam])
    o = oracle.render(sc.octrees, sc.poses, cam, oracle.Opts(1, 1e-4))
    im = lambda x, c=None: split_images(x.cpu().numpy(), [cam], c)[0]
    check_forward(im(rgb, 3), im(depth), im(alpha), o[0], o[1], o[2], f"{n} voxels")


# three and nine views, with voxels below the projection's queue and with enough of them for groups of eight views (nine:
# a group and a remainder), in which a warp tests the box around its leaves first, on leaves in order, out of order and
# with warps that hold leaves of two octrees: the images of each view alone, bit for bit
@pytest.mark.gpu
@pytest.mark.parametrize("n_view,shuffle,n", [(3, False, 40003), (3, True, 40003), (9, False, 40003),
                                              (3, False, 1670003), (3, True, 1670003), (9, False, 556003)])
def test_projection_of_several_views(dv, n_view, shuffle, n):
    rng = np.random.default_rng(n_view)
    key = _grid(6 if n < 64 ** 3 else 7, 0.0, rng, n)
    octs = [_octree(key[rng.permutation(key.size)] if shuffle else key, 0.5, rng, 8.0)]
    octs += [_octree(_grid(3, 0.0, rng, 77), 2.0, rng, 1.0, synth.ACTOR, (0.4, 0.45, 0.3)) for _ in range(2)]
    poses = [synth.Pose()] + [synth.Pose(synth.random_rotation(rng), rng.uniform(-2, 2, 3)) for _ in range(2)]
    cams = [synth.pinhole(35, 19, 50.0, synth.Pose(synth.random_rotation(rng), rng.uniform(-3, 3, 3)), 0.05, 4.0)
            for _ in range(n_view)]
    ds = device_scene(synth.Scene(octs, poses))
    assert n_view * sum(o.n for o in octs) < 400000 if n == 40003 else n_view * sum(o.n for o in octs) >= 5000000
    both = gpu_render(ds, poses, cams)[:3]
    for c, cam in enumerate(cams):
        for a, b in zip(both, gpu_render(ds, poses, [cam])[:3]):
            n = cam.W * cam.H
            np.testing.assert_array_equal(a[c * n:(c + 1) * n].cpu().numpy(), b.cpu().numpy())


def _keys_t(keys):
    import torch
    return torch.as_tensor(np.asarray(keys, np.uint64).view(np.int64), device="cuda")


def _check_corners(dv, keys, level):
    grid, index = dv.dv_shared_corners(_keys_t(keys), level)
    pts = oi.corner_grid_points(keys, level).reshape(-1, 3).astype(np.uint64)
    packed = (pts[:, 2] << np.uint64(42)) | (pts[:, 1] << np.uint64(21)) | pts[:, 0]
    ref, inv = np.unique(packed, return_inverse=True)
    np.testing.assert_array_equal(grid.cpu().numpy().view(np.uint64), ref)
    np.testing.assert_array_equal(index.cpu().numpy().astype(np.int64).ravel(), inv.ravel())


# the sort of 8 n corners just below and above the counted sort's first size, and far above it (a ragged last tile)
@pytest.mark.gpu
@pytest.mark.parametrize("over", [0, 1, 120011])
@pytest.mark.parametrize("max_level", [6, 15])
def test_counted_sort(dv, over, max_level):
    import torch
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    n = 16 * 256 * n_sm // 8 + over
    rng = np.random.default_rng(over)
    keys = _grid(6, 0.0, rng, n)
    _check_corners(dv, keys[rng.permutation(n)], max_level)


@pytest.mark.gpu
def test_corners_of_leaves_outside_the_root(dv):
    # an index beyond its level's grid is a point like any other (coordinates of up to 21 bits)
    keys = synth.pack_keys([3, 3, 2, 0, 3], [7, 8, 5, 1, 300], [0, 15, 4, 0, 2], [7, 9, 2, 3, 70])
    _check_corners(dv, keys, 3)


# exact ties, points a few 1e-7 of the distance apart, repeated points and points that are not numbers, near the
# origin and (coordinates of thousands, leaves of centimetres) far from it
@pytest.mark.gpu
@pytest.mark.parametrize("center,root", [((0.0, 0.0, 0.0), 2.0), ((4000.5, -2500.25, 80.0), 3.7)])
def test_soft_prior_ties(dv, center, root):
    import torch
    rng = np.random.default_rng(5)
    L = 5
    keys = _grid(L, 0.3, rng)
    s = root / 2 ** L
    pts, _ = oi.shared_corners(keys, L)
    world = oi.grid_to_world(pts, center, root, L)
    at = world[rng.choice(len(world), 150)]
    d = rng.normal(size=at.shape) * s
    cloud = np.concatenate([at + d, at - d, at + d[:, [1, 2, 0]], at + d * (1 + 3e-7), at + d, at[:5],
                            np.asarray(center) + rng.uniform(-0.5, 0.5, (200, 3)) * root])
    cloud = np.float32(cloud[rng.permutation(len(cloud))])
    ref = oi.soft_prior(oi.nearest_distance(world, np.float64(cloud)), s)
    bad = np.float32([[np.nan, 0, 0], [np.inf, -np.inf, 0], [1e30, 1e30, -1e30]])
    grid, _ = dv.dv_shared_corners(_keys_t(keys), L)
    for c in (cloud, np.concatenate([bad, cloud, bad])):
        dens = dv.dv_soft_prior(grid, center, root, L, torch.as_tensor(c, device="cuda"), s).cpu().numpy()
        np.testing.assert_allclose(dens, ref, rtol=0, atol=1e-5)


def _reached(keys, center, root, cloud, thr):
    """The leaves of the subdivision's definition in FP64: those among the cells floor((p - thr) / s) to
    floor((p + thr) / s) of a point p whose box is within thr of it.  It is the oracle's set, except that a leaf
    whose upper face is at exactly thr is not among the cells."""
    lev, *ijk = oi._unpack(keys)
    s = root / 2.0 ** lev
    hit = np.zeros(len(keys), bool)
    for p in np.float64(cloud) - (np.asarray(center, np.float64) - 0.5 * root):
        near, d2 = np.ones(len(keys), bool), np.zeros(len(keys))
        for a in range(3):
            near &= (ijk[a] >= np.floor((p[a] - thr) / s)) & (ijk[a] <= np.floor((p[a] + thr) / s))
            d2 += np.maximum(np.maximum(ijk[a] * s - p[a], 0.0), p[a] - (ijk[a] * s + s)) ** 2
        hit |= near & (d2 <= thr * thr)
    return hit


# thresholds far below a leaf (every distance in FP64), of a leaf's size (also met exactly, in numbers that are
# exact in both arithmetics) and beyond the root
@pytest.mark.gpu
@pytest.mark.parametrize("center,root,thr", [((0.0, 0.0, 0.0), 2.0, 1e-7), ((0.0, 0.0, 0.0), 2.0, 0.125),
                                             ((0.0, 0.0, 0.0), 2.0, 5.0), ((310.1, -77.7, 12.9), 2.3, 0.11)])
def test_subdivide_thresholds(dv, center, root, thr):
    import torch
    rng = np.random.default_rng(6)
    keys = np.concatenate([_grid(3, 0.5, rng), _grid(4, 0.05, rng), _grid(1, 0.4, rng)])
    keys = keys[rng.permutation(keys.size)]
    cloud = np.asarray(center) + rng.uniform(-0.7, 0.7, (20, 3)) * root
    if root == 2.0:
        cloud = np.concatenate([cloud, rng.integers(-8, 9, (10, 3)) / 8.0, rng.integers(-17, 18, (10, 3)) / 16.0])
    cloud = np.float32(cloud)
    thr = float(np.float32(thr))
    out = dv.dv_subdivide_round(_keys_t(keys), 4, center, root, torch.as_tensor(cloud, device="cuda"), thr)
    hit = _reached(keys, center, root, cloud, thr)
    split = oi.subdivide_round(keys, center, root, cloud, thr)[1]
    assert hit.any() and not (hit & ~split).any() and ((hit == split).all() or thr == 0.125)
    lev, i, j, k = (x[hit] for x in oi._unpack(keys))
    ref = np.concatenate([keys[~hit]] + [oi._pack(lev + 1, 2 * i + (c & 1), 2 * j + (c >> 1 & 1), 2 * k + (c >> 2))
                                         for c in range(8)])
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), ref)


# a threshold of more than 1e9 cells of the finest level, and a point nearly as far away: every leaf is within it
@pytest.mark.gpu
def test_subdivide_threshold_of_many_roots(dv):
    import torch
    keys = np.concatenate([_grid(l, 2.0, np.random.default_rng(l)) for l in (1, 2, 3)])
    center, root, thr = (0.0, 0.0, 0.0), 1.1, 5000.0
    cloud = torch.tensor([[-4196.0, 0.0, 0.0]], device="cuda")
    out = dv.dv_subdivide_round(_keys_t(keys), 3, center, root, cloud, thr)
    assert _reached(keys, center, root, cloud.cpu().numpy(), thr).all()
    assert out.numel() == 8 * keys.size


# thresholds of several leaves, at which leaves look for points (beside coarse leaves that points look for): a cluster in
# a corner whose reach ends inside the set, exact ties, equal keys (the first counts), a leaf outside the grid, points
# that are not numbers; far from the origin; more of the points' cells than are looked into; and cells of which a point
# has 7e13 in reach
@pytest.mark.gpu
@pytest.mark.parametrize("center,root,thr,levels", [((0.0, 0.0, 0.0), 2.0, 0.5, (1, 3, 5, 6)),
                                                    ((4000.5, -2500.25, 80.0), 3.7, 0.61, (2, 6)),
                                                    ((0.0, 0.0, 0.0), 2.0, 300.0, (1, 4, 7)),
                                                    ((1.0, 2.0, 3.0), 10.0, 3.0, (2, 9, 16))])
def test_subdivide_reach_of_many_leaves(dv, center, root, thr, levels):
    import torch
    rng = np.random.default_rng(9)
    parts = []
    for l in levels:
        m = 1 << l
        c = rng.integers(0, m, (min(600, m ** 3), 3))
        parts.append(np.unique(synth.pack_keys(np.full(len(c), l), *c.T)))
    keys = np.concatenate(parts)
    keys = keys[rng.permutation(keys.size)]
    L = levels[-1]
    keys = np.concatenate([keys, synth.pack_keys([L, L], [1 << L, 3], [0, 5], [1, 2 << L]), keys[:40]])
    corner = np.asarray(center) - 0.4 * root
    cloud = corner + rng.uniform(-0.15, 0.1, (60, 3)) * root
    if root == 2.0:
        cloud = np.concatenate([cloud, corner.round(1) + rng.integers(-3, 4, (20, 3)) / 16.0])
    cloud = np.float32(np.concatenate([cloud, cloud[:5]]))
    thr = float(np.float32(thr))
    bad = np.float32([[np.nan, 0, 0], [np.inf, 0, 0], [1e30, -1e30, 0]])
    out = dv.dv_subdivide_round(_keys_t(keys), L, center, root, torch.as_tensor(np.concatenate([bad, cloud]), device="cuda"), thr)
    lev, *ijk = oi._unpack(keys)
    first = np.zeros(keys.size, bool)
    first[np.unique(keys, return_index=True)[1]] = True
    hit = _reached(keys, center, root, cloud, thr) & first & (np.stack(ijk, 1) < (1 << lev)[:, None]).all(1)
    assert hit.any() and ((~hit & first).sum() > 50 or thr > root)
    lev, i, j, k = (x[hit] for x in oi._unpack(keys))
    ref = np.concatenate([keys[~hit]] + [oi._pack(lev + 1, 2 * i + (c & 1), 2 * j + (c >> 1 & 1), 2 * k + (c >> 2))
                                         for c in range(8)])
    np.testing.assert_array_equal(out.cpu().numpy().view(np.uint64), ref)


def _crowded(candidates):
    """100 keys whose homes in the hash tables of 2^10 to 2^13 slots (unsalted) are the same slot each."""
    with np.errstate(over="ignore"):
        h = candidates ^ (candidates >> np.uint64(32))
        h = h * np.uint64(0x9e3779b97f4a7c15)
        h = (h ^ (h >> np.uint64(29))) * np.uint64(0x9e3779b97f4a7c15)
    home = (h >> np.uint64(51)).astype(np.int64)
    return candidates[home == np.bincount(home).argmax()][:100]


# keys that find no slot within the probes of their home in any unsalted table: leaf keys of the subdivision, cells of
# the prior's points
@pytest.mark.gpu
def test_crowded_hash_tables(dv):
    import torch
    rng = np.random.default_rng(12)
    L, center, root = 12, (0.0, 0.0, 0.0), 4096.0
    c = rng.integers(0, 1 << L, (1 << 20, 3))
    keys = _crowded(np.unique(synth.pack_keys(np.full(len(c), L), *c.T)))
    _, *ijk = oi._unpack(keys)
    centres = np.stack(ijk, 1) + 0.5 - 2048.0
    assert len(keys) == 100
    cloud = torch.as_tensor(np.float32(centres[::2]), device="cuda")
    out = dv.dv_subdivide_round(_keys_t(keys), L, center, root, cloud, 0.25)
    hit = _reached(keys, center, root, centres[::2], 0.25)
    assert hit[::2].all()
    np.testing.assert_array_equal(out[:(~hit).sum()].cpu().numpy().view(np.uint64), keys[~hit])
    assert out.numel() == (~hit).sum() + 8 * hit.sum()
    # cells of the points at s_min = 1 / 3: the finest cells, offset by 2^20
    cell = np.unique(np.concatenate([(z + (1 << 20) << 42) | (y + (1 << 20) << 21) | (x + (1 << 20))
                                     for x, y, z in [rng.integers(0, 1 << L, (3, 1 << 20))]]).astype(np.uint64))
    cell = _crowded(cell).astype(np.int64)
    assert len(cell) == 100
    at = np.stack([cell & 0x1fffff, (cell >> 21) & 0x1fffff, cell >> 42], 1) - (1 << 20)
    s = float(np.float32(1.0 / 3.0))
    pts = np.float32(at + 0.5 - 2048.0)
    grid, _ = dv.dv_shared_corners(_keys_t(synth.pack_keys(np.full(100, L), *at.T)), L)
    dens = dv.dv_soft_prior(grid, center, root, L, torch.as_tensor(pts, device="cuda"), s).cpu().numpy()
    p, _ = oi.shared_corners(synth.pack_keys(np.full(100, L), *at.T), L)
    ref = oi.soft_prior(oi.nearest_distance(oi.grid_to_world(p, center, root, L), np.float64(pts)), s)
    np.testing.assert_allclose(dens, ref, rtol=0, atol=1e-5)


@pytest.mark.gpu
def test_visibility_many_cameras(dv):
    # cameras all around, inside and outside the root, with narrow and wide views; a ragged last block
    rng = np.random.default_rng(8)
    keys = np.concatenate([_grid(4, 0.0, rng, 1500), _grid(2, 0.5, rng)])
    center, root = (0.0, 0.0, 4.0), 16.0
    for n_cam in (1, 2, 12):
        cams = [synth.pinhole(64, 48, float(rng.uniform(5, 60)),
                              synth.Pose(synth.random_rotation(rng), rng.uniform(-7, 7, 3)),
                              float(rng.uniform(0.05, 2.0)), float(rng.uniform(3.0, 8.0))) for _ in range(n_cam)]
        out = dv.dv_visibility_prune(_keys_t(keys), 4, center, root, cams, z_min=-2.0).cpu().numpy().view(np.uint64)
        keep = oi.visible_from(keys, center, root, cams, -2.0)
        assert 0 < keep.sum() < len(keys)
        np.testing.assert_array_equal(out, keys[keep])


# maps of one texel (all lanes in one cell), of a few, and finer than the pixels; a ragged last warp
@pytest.mark.gpu
@pytest.mark.parametrize("He,We", [(1, 1), (3, 5), (64, 128)])
def test_sky_shared_cells(dv, He, We):
    import torch
    rng = np.random.default_rng(He)
    cam = synth.pinhole(37, 21, 75.0, synth.look_at((0.0, 0.0, 0.0), (-1.0, 0.1, 0.3)), 0.05, 50.0)
    P = cam.W * cam.H
    env = rng.uniform(0, 1, (He, We, 3)).astype(np.float32)
    alpha = rng.uniform(0, 1, P).astype(np.float32)
    g = np.float32(rng.normal(size=(P, 3)))
    g[rng.uniform(size=P) < 0.2] = 0.0
    t = lambda a: torch.as_tensor(a, device="cuda")
    d_env, d_alpha = torch.zeros((He, We, 3), device="cuda"), torch.zeros(P, device="cuda")
    dv.dv_sky_backward([cam], t(env), t(alpha), t(g), d_env, d_alpha)
    torch.cuda.synchronize()
    ref_env, ref_alpha, _ = osky.backward(alpha, osky.pixel_directions(cam), env, np.float64(g))
    for a, b in ((d_env, ref_env), (d_alpha, ref_alpha)):  # the bound of the sky's parity tests
        lim = 1e-5 * (np.abs(b) + np.abs(b).max()) + 1e-7
        assert (np.abs(a.cpu().numpy() - b) <= lim).all()


@pytest.mark.gpu
def test_gradients_have_storage_of_their_own(dv):
    # dropping one octree's gradient frees it, saving one writes it alone
    rng = np.random.default_rng(2)
    octs = [_octree(_grid(2, 0.5, rng), 1.0, rng, 2.0)]
    octs += [_octree(_grid(2, 0.5, rng), 1.0, rng, 0.5, synth.ACTOR, (0.25, 0.25, 0.25)) for _ in range(2)]
    ds = device_scene(synth.Scene(octs, [synth.Pose()] * 3))
    ts = [t.requires_grad_() for o in ds for t in (o.dens, o.sh)]
    out = dv.render(ds, [synth.Pose()] * 3, [orbit(9, 7, 40.0, 20.0)])
    sum(x.sum() for x in out).backward()
    assert len({t.grad.untyped_storage().data_ptr() for t in ts}) == len(ts)
    assert all(t.grad.untyped_storage().nbytes() == 4 * t.numel() for t in ts)


def _side_path(idx, level, X, Lk):
    """The projection's closed form of one axis of the depth-order path (32-bit arithmetic)."""
    mask = (1 << level) - 1
    if X < 0:
        return idx
    if X >> (Lk + 1):
        return ~idx & mask
    cell = X >> (Lk + 1 - level)
    diff = idx ^ cell
    if diff == 0:
        return 0
    top = diff.bit_length() - 1
    return (1 << top) | ((~idx if (cell >> top) & 1 else idx) & ((1 << top) - 1))


# the device's depth order, through images that depend on it: leaves of four levels, cameras on the planes of nodes of
# several levels, on a face and a corner of the root, inside leaves and outside the root on either side of each axis
@pytest.mark.gpu
@pytest.mark.parametrize("eye", [(0.0, 0.0, 0.0), (0.25, -0.5, 0.125), (0.5, 0.0625, -0.75), (0.11, -0.23, 0.37),
                                 (-1.0, 0.3, 0.0), (1.0, 1.0, -1.0), (1.75, -1.5, 1.25), (-2.0, 0.25, 0.5)])
def test_depth_order(dv, eye):
    rng = np.random.default_rng(21)
    i, j, k = np.unravel_index(np.arange(8), (2, 2, 2))
    keys = []
    for level in (1, 2, 3, 4):  # most of a level's cells are split further
        split = rng.uniform(size=i.size) < (0.0 if level == 4 else 0.8)
        keys.append(synth.pack_keys(np.full((~split).sum(), level), i[~split], j[~split], k[~split]))
        c = np.arange(8)
        i, j, k = ((2 * x[split][:, None] + (c >> n & 1)).ravel() for n, x in ((0, i), (1, j), (2, k)))
    key = np.concatenate(keys)
    sc = synth.Scene([_octree(key[rng.permutation(key.size)], 1.0, rng, 2.0, degree=0)], [synth.Pose()])
    for at in ((0.05, 0.1, -0.2), (0.9, -0.7, 0.3)):
        cam = synth.pinhole(31, 23, 70.0, synth.look_at(eye, at), 0.02, 20.0)
        rgb, depth, alpha, _ = gpu_render(device_scene(sc), sc.poses, [cam], eps=0.0)
        o = oracle.render(sc.octrees, sc.poses, cam, oracle.Opts(1, 0.0))
        im = lambda x, c=None: split_images(x.cpu().numpy(), [cam], c)[0]
        check_forward(im(rgb, 3), im(depth), im(alpha), o[0], o[1], o[2], f"eye {eye}")


# (the formula alone, in Python; test_depth_order has the kernel)
@pytest.mark.parametrize("Lk", [0, 1, 4])
def test_depth_path_closed_form(Lk):
    # node by node: at each node on the way to the leaf, the bit is flipped where the camera lies on the positive
    # side of the node's plane (its coordinate on the lattice of half cells, on a plane: not below it)
    for level in range(Lk + 1):
        for idx in range(1 << level):
            for X in range(-3, (2 << Lk) + 4):
                path = 0
                for d in range(level):
                    node = idx >> (level - d)
                    plane = (2 * node + 1) << (Lk - d)
                    bit = (idx >> (level - d - 1)) & 1
                    path = 2 * path + (bit ^ (1 if X >= plane else 0))
                assert _side_path(idx, level, X, Lk) == path, (level, idx, X)
