"""The shaft walk (the default accumulation kernel) against the per-ray walk (GM_F_FIX_L1) on the same
scenes: both decide every ray with the same arithmetic and add the weights in the same order, so the
maps are equal bit for bit. Sizes at the edges of a warp tile, of a fill step (512 fixations), of a batch
and of the ranges of the block sizes (456 tiles, 256 fixations, a quarter as many fixations as tiles);
sample sets of 393216 samples and more, which have tiles of 128 samples where those lie on few triangles,
with such tiles in the majority and without any, near a surface, over the budget, reached by few fixations
and in a posed scene; trees of one and two triangles; triangles far smaller than the sample spacing (a
shaft over its budget); an eye close to the surface, whose rays differ in
their dominant axis and cross the planes through the eye."""
import math

import numpy as np
import pytest

from synth import meshes as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_07571_gb300 import build
    build.build()
    import paper_2601_07571_gb300 as G
    ctx = G.gm_create(0)
    yield G, ctx
    G.gm_destroy(ctx)


def _scene(kind):
    """(vertices, indices) of one mesh."""
    tri = np.array([[0.0, 0.0, 1.0], [0.6, 0.0, 1.0], [0.0, 0.6, 1.0]], np.float32)
    if kind == "one":
        return tri, np.array([[0, 1, 2]], np.uint32)
    if kind == "two":
        return np.concatenate([tri, tri + np.float32([0.1, 0.1, -0.3])]), np.array([[0, 1, 2], [3, 4, 5]], np.uint32)
    if kind == "fine":      # 80k triangles of about 1 mm on a 6 cm sphere, before a coarse one
        v, f = M.uv_sphere(12, 24, 0.5)
        return M.merge([M.uv_sphere(142, 284, 0.06, 0.05, 30.0, seed=3), (M.translate(v, (0.0, 0.0, 0.9)), f)])
    if kind == "mixed":     # a box of large triangles (seven tenths of the samples) beside a sphere of small ones
        v, f = M.uv_sphere(60, 120, 0.4, 0.05, 6.0, seed=4)
        return M.merge([M.box((0.0, 0.0, 0.0), 0.8), (M.translate(v, (0.0, 0.3, 1.5)), f)])
    return M.uv_sphere(40, 80, 1.0, 0.1, 4.0, seed=5)


def _points(kind, v, f, n, rng):
    t = v[f.astype(np.int64)].astype(np.float64)
    tri = rng.integers(0, len(f), n)
    if kind == "mixed":
        tri[rng.random(n) < 0.7] %= 12
    s, u = np.sqrt(rng.random((n, 1))), rng.random((n, 1))
    p = (1 - s) * t[tri, 0] + s * (1 - u) * t[tri, 1] + s * u * t[tri, 2]
    return np.ascontiguousarray(p, np.float32), tri.astype(np.uint32)


@pytest.mark.parametrize("kind,n,nf,theta,near,windows", [
    ("one", 1, 3, 4.0, False, 1), ("two", 33, 40, 4.0, False, 1),
    ("sphere", 31, 511, 2.0, False, 1), ("sphere", 32, 512, 2.0, False, 3), ("sphere", 1000, 1300, 6.0, False, 5),
    ("sphere", 14592, 255, 2.0, False, 1), ("sphere", 14592, 256, 2.0, False, 2), ("sphere", 14624, 256, 2.0, False, 1),
    ("sphere", 32768, 256, 2.0, False, 1), ("sphere", 32769, 256, 2.0, False, 1),
    ("mixed", 65537, 300, 2.0, False, 1), ("mixed", 70001, 300, 3.0, False, 3),
    ("mixed", 393215, 60, 2.0, False, 1), ("mixed", 393216, 60, 2.0, False, 1), ("mixed", 393301, 60, 3.0, False, 3),
    ("fine", 2048, 600, 1.0, False, 1), ("fine", 65600, 60, 1.0, False, 1), ("fine", 393300, 20, 1.0, False, 1), ("sphere", 3000, 200, 15.0, True, 1), ("sphere", 257, 0, 1.0, False, 2)])
def test_shaft_walk_equals_per_ray_walk(env, kind, n, nf, theta, near, windows):
    G, ctx = env
    rng = np.random.default_rng(n + nf)
    v, f = _scene(kind)
    scene = G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)])
    xyz, tri = _points(kind, v, f, n, rng)
    samples = G.gm_samples_from_points(scene, xyz, tri)
    at = xyz[rng.integers(0, n, nf)].astype(np.float64)
    if near:      # a few centimetres off the surface, looking along it or at it
        eye = at * (1.0 + 0.03 * rng.random((nf, 1)))
        gaze = rng.normal(size=(nf, 3))
    else:
        eye = rng.normal(size=(nf, 3))
        eye *= 2.5 / np.maximum(np.linalg.norm(eye, axis=1, keepdims=True), 1e-9)
        gaze = at - eye
    fix = [np.ascontiguousarray(eye, np.float32), np.ascontiguousarray(gaze, np.float32),
           rng.uniform(0.1, 0.6, nf).astype(np.float32), np.sort(rng.uniform(0.0, windows, nf))]
    out = []
    for flags in (0, G.GM_F_FIX_L1):
        kw = dict(t_begin=0.0, t_end=float(windows), window_s=1.0) if windows > 1 else {}
        m = G.gm_accumulate_fixations(scene, samples, *fix, G.make_params(math.radians(theta), normalize=False, flags=flags, **kw))
        W, ns, st, _ = G.gm_map_info(m)
        maps = np.empty((W, ns), np.float32)
        top = [G.gm_map_copy(m, w, maps[w]) for w in range(W)]
        G.gm_map_free(m)
        # the cone tests evaluated depend on the size of a form's tiles: between the in-cone and all pairs
        assert st["in_cone"] <= st["pairs_tested"] <= st["pairs"]
        out.append((maps, top, {k: st[k] for k in ("pairs", "in_cone", "visible")}))
    G.gm_samples_free(samples)
    G.gm_scene_free(scene)
    assert W == windows and out[0][2] == out[1][2] and out[0][1] == out[1][1]
    assert np.array_equal(out[0][0], out[1][0])
    if nf > 10:
        assert out[0][2]["visible"] > 0


def _floor(n, occluder):
    """n samples on a grid of a unit floor of two triangles (so that every tile of 128 is wide), the occluder's
    triangles after it; samples lie on floats, so that an eye can stand exactly above one."""
    q = np.array([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0], [1.0, 0.0, 1.0], [0.0, 0.0, 1.0]], np.float32)
    v, f = M.merge([(q, np.array([[0, 2, 1], [0, 3, 2]], np.uint32)), occluder])
    k = math.ceil(math.sqrt(n))
    x, z = np.divmod(np.arange(n), k)
    xyz = np.ascontiguousarray(np.stack([(x + 0.5) / k, np.zeros(n), (z + 0.5) / k], 1), np.float32)
    return v, f, xyz, (xyz[:, 2] > xyz[:, 0]).astype(np.uint32)


def test_wide_tile_with_a_ray_in_a_coordinate_plane(env):
    """Eyes exactly above samples, 6 mm over the floor: the ray straight down has no image point on the side of the
    tile's first ray (0 / 0 there), and what hides it crosses the plane through the eye."""
    G, ctx = env
    rng = np.random.default_rng(5)
    q = np.array([[0.2, 0.003, 0.2], [0.8, 0.003, 0.2], [0.8, 0.003, 0.8], [0.2, 0.003, 0.8]], np.float32)
    v, f, xyz, tri = _floor(400000, (q, np.array([[0, 2, 1], [0, 3, 2]], np.uint32)))
    nf = 400
    at = rng.integers(0, len(xyz), nf)
    turn = rng.uniform(0.0, 2.0 * math.pi, nf)
    tilt = math.radians(24.0)
    eye = xyz[at] + np.float32([0.0, 0.006, 0.0])
    gaze = np.stack([math.sin(tilt) * np.cos(turn), np.full(nf, -math.cos(tilt)), math.sin(tilt) * np.sin(turn)], 1)
    fix = [np.ascontiguousarray(eye, np.float32), np.ascontiguousarray(gaze, np.float32),
           rng.uniform(0.1, 0.6, nf).astype(np.float32), np.arange(float(nf))]
    scene = G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)])
    samples = G.gm_samples_from_points(scene, xyz, tri)
    out = []
    for flags in (0, G.GM_F_FIX_L1):
        m = G.gm_accumulate_fixations(scene, samples, *fix, G.make_params(math.radians(9.0), normalize=False, flags=flags))
        _, ns, st, _ = G.gm_map_info(m)
        values = np.empty(ns, np.float32)
        G.gm_map_copy(m, 0, values)
        G.gm_map_free(m)
        out.append((values, st["in_cone"], st["visible"]))
    G.gm_samples_free(samples)
    G.gm_scene_free(scene)
    assert out[0][1:] == out[1][1:] and 0 < out[0][2] < out[0][1]
    assert np.array_equal(out[0][0], out[1][0])


def _maps(G, scene, samples, fix, theta, flags, **kw):
    m = G.gm_accumulate_fixations(scene, samples, *fix, G.make_params(theta, normalize=False, flags=flags, **kw))
    W, ns, st, _ = G.gm_map_info(m)
    values = np.empty((W, ns), np.float32)
    for w in range(W):
        G.gm_map_copy(m, w, values[w])
    G.gm_map_free(m)
    return values, st["in_cone"], st["visible"]


@pytest.mark.parametrize("n,nf,theta,windows", [
    (1 << 19, 1, 1.0, 1), (1 << 19, 40, 1.0, 3), ((1 << 19) + 77, 2048, 0.3, 5), (1 << 19, 2048, 2.0, 1),
    ((1 << 19) - 1, 40, 1.0, 1), (1 << 19, 2049, 0.3, 2)])
def test_blocks_of_wide_tiles(env, n, nf, theta, windows):
    """Sets of 2^19 samples and more whose tiles few fixations reach take smaller blocks, by a probe on the device
    that lists of up to 2048 fixations get: either way the per-ray walk's maps."""
    G, ctx = env
    rng = np.random.default_rng(nf)
    ball = M.uv_sphere(30, 60, 0.1, 0.1, 8.0, seed=2)
    v, f, xyz, tri = _floor(n, (M.translate(ball[0], (0.5, 0.2, 0.5)), ball[1]))
    at = xyz[rng.integers(0, n, nf)].astype(np.float64)
    eye = np.stack([rng.uniform(0, 1, nf), rng.uniform(0.4, 0.8, nf), rng.uniform(0, 1, nf)], 1)
    fix = [np.ascontiguousarray(eye, np.float32), np.ascontiguousarray(at - eye, np.float32),
           rng.uniform(0.1, 0.6, nf).astype(np.float32), rng.uniform(0, windows, nf)]
    kw = dict(t_begin=0.0, t_end=float(windows), window_s=1.0) if windows > 1 else {}
    scene = G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)])
    samples = G.gm_samples_from_points(scene, xyz, tri)
    a, b = (_maps(G, scene, samples, fix, math.radians(theta), flags, **kw) for flags in (0, G.GM_F_FIX_L1))
    G.gm_samples_free(samples)
    G.gm_scene_free(scene)
    assert a[1:] == b[1:] and a[2] > 0 and np.array_equal(a[0], b[0])


@pytest.mark.parametrize("n,nf", [(7000, 100), (7000, 400), (14592, 300), (20000, 6000), (130000, 60), (400000, 50)])
def test_pair_records_of_every_block_size(env, n, nf):
    """The recorded pairs (blocks of 512, 1024, 1024, 512 and 256 threads; 256 with wide tiles) are the per-ray walk's:
    sample, fixation, visibility and weight."""
    G, ctx = env
    rng = np.random.default_rng(n)
    v, f = _scene("mixed" if n == 400000 else "sphere")
    xyz, tri = _points("mixed" if n == 400000 else "sphere", v, f, n, rng)
    eye = rng.normal(size=(nf, 3))
    eye *= 2.5 / np.linalg.norm(eye, axis=1, keepdims=True)
    at = xyz[rng.integers(0, n, nf)].astype(np.float64)
    fix = [np.ascontiguousarray(eye, np.float32), np.ascontiguousarray(at - eye, np.float32),
           rng.uniform(0.1, 0.6, nf).astype(np.float32), np.arange(float(nf))]
    scene = G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)])
    samples = G.gm_samples_from_points(scene, xyz, tri)
    cap, out = 8_000_000, []
    for flags in (0, G.GM_F_FIX_L1):
        m = G.gm_accumulate_fixations(scene, samples, *fix, G.make_params(
            math.radians(0.6), normalize=False, flags=flags | G.GM_F_DEBUG_PAIRS, debug_pair_cap=cap))
        p = G.gm_map_debug_pairs(m, cap)
        G.gm_map_free(m)
        order = np.argsort(p["sample"].astype(np.int64) * (1 << 20) + p["fix"])
        out.append([p[k][order] for k in ("sample", "fix", "visible", "g")])
    G.gm_samples_free(samples)
    G.gm_scene_free(scene)
    assert 0 < len(out[0][0]) < cap
    assert all(np.array_equal(a, b) for a, b in zip(*out))


def _above(n, rng, lo=0.3, hi=0.6, target=None):
    """n viewers above the unit floor, gazing at points of it (or at one point)."""
    eye = np.stack([rng.uniform(0, 1, n), rng.uniform(lo, hi, n), rng.uniform(0, 1, n)], 1)
    at = np.stack([rng.uniform(0, 1, n), np.zeros(n), rng.uniform(0, 1, n)], 1) if target is None else np.float64(target)
    return [np.ascontiguousarray(eye, np.float32), np.ascontiguousarray(at - eye, np.float32),
            rng.uniform(0.1, 0.6, n).astype(np.float32)]


def test_wide_tiles_over_the_budget(env):
    """320k triangles of about half a millimetre between the viewers and a floor in wide tiles: shafts run over their budget and
    their four rays a lane walk the tree one by one."""
    G, ctx = env
    rng = np.random.default_rng(8)
    ball = M.uv_sphere(284, 568, 0.06, 0.05, 30.0, seed=3)
    v, f, xyz, tri = _floor(400000, (M.translate(ball[0], (0.5, 0.07, 0.5)), ball[1]))
    fix = [*_above(60, rng, target=(0.52, 0.02, 0.5)), np.arange(60.0)]
    scene = G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)])
    samples = G.gm_samples_from_points(scene, xyz, tri)
    a, b = (_maps(G, scene, samples, fix, math.radians(2.0), flags) for flags in (0, G.GM_F_FIX_L1))
    G.gm_samples_free(samples)
    G.gm_scene_free(scene)
    assert a[1:] == b[1:] and 0 < a[2] < a[1] and np.array_equal(a[0], b[0])


@pytest.mark.parametrize("density,nf", [(400000.0, 300), (530000.0, 45)])
def test_wide_tiles_of_a_posed_scene(env, density, nf):
    """A floor in wide tiles (whole blocks; halves of blocks), turning, below a ball that moves: every window's map is
    the per-ray walk's."""
    G, ctx = env
    rng = np.random.default_rng(9)
    q = np.array([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0], [1.0, 0.0, 1.0], [0.0, 0.0, 1.0]], np.float32)
    ball, windows = M.uv_sphere(30, 60, 0.12, 0.1, 8.0, seed=2), 3
    scene = G.gm_build_scene(ctx, [(q, np.array([[0, 2, 1], [0, 3, 2]], np.uint32), np.eye(4), 0), (*ball, np.eye(4), 1)],
                             dynamic=True)
    samples = G.gm_sample_surface(scene, [density, 0.0], 3)
    poses = np.tile(np.eye(4), (windows, 2, 1, 1))
    for w in range(windows):
        a = 0.1 * w
        poses[w, 0, :3, :3] = [[math.cos(a), 0, math.sin(a)], [0, 1, 0], [-math.sin(a), 0, math.cos(a)]]
        poses[w, 1, :3, 3] = [0.3 + 0.2 * w, 0.2, 0.5]
    fix = [*_above(nf, rng), np.sort(rng.uniform(0, windows, nf))]
    prm = dict(t_begin=0.0, t_end=float(windows), window_s=1.0, normalize=False)
    out = []
    for flags in (0, G.GM_F_FIX_L1):
        m = G.gm_accumulate_dynamic(scene, samples, *fix, G.make_params(math.radians(2.0), flags=flags, **prm), poses)
        W, ns, st, _ = G.gm_map_info(m)
        values = np.empty((W, ns), np.float32)
        for w in range(W):
            G.gm_map_copy(m, w, values[w])
        G.gm_map_free(m)
        out.append((values, st["in_cone"], st["visible"]))
    G.gm_samples_free(samples)
    G.gm_scene_free(scene)
    assert out[0][1:] == out[1][1:] and 0 < out[0][2] < out[0][1]
    assert np.array_equal(out[0][0], out[1][0]) and (out[0][0] > 0).any(1).all()
