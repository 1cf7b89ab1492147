"""The scene build and the sorts at the sizes where their forms change: trees of a few triangles, of one
block's clustering (1024 clusters), of several blocks, with every neighbour radius -- the maps traced
through them equal those of the other builder's tree bit for bit -- and fixation lists around the
one-block sort (2048), whose windows equal single calls over each window's interval."""
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


def _soup(n, rng):
    """n small triangles on a noisy sphere."""
    c = rng.normal(size=(n, 3))
    c /= np.linalg.norm(c, axis=1, keepdims=True)
    v = c[:, None, :] * rng.uniform(0.7, 1.0, (n, 1, 1)) + rng.normal(scale=0.15, size=(n, 3, 3))
    return np.ascontiguousarray(v.reshape(-1, 3), np.float32), np.arange(3 * n, dtype=np.uint32).reshape(-1, 3)


def _look(n, rng):
    eye = rng.normal(size=(n, 3))
    eye *= 3.0 / np.linalg.norm(eye, axis=1, keepdims=True)
    return (np.ascontiguousarray(eye, np.float32), np.ascontiguousarray(-eye + rng.normal(scale=0.4, size=(n, 3)), np.float32),
            rng.uniform(0.1, 0.6, n).astype(np.float32))


def _map(G, scene, samples, fix, ts, **kw):
    m = G.gm_accumulate_fixations(scene, samples, *fix, ts, G.make_params(math.radians(2.0), normalize=False, **kw))
    W, ns, st, _ = G.gm_map_info(m)
    out = np.empty((W, ns), np.float32)
    for w in range(W):
        G.gm_map_copy(m, w, out[w])
    G.gm_map_free(m)
    return out, st


@pytest.mark.parametrize("n,radius", [(2, 0), (3, 4), (31, 0), (1024, 0), (1025, 0), (1537, 64), (2049, 16), (5000, 32),
                                      (70000, 0)])
def test_clustered_tree_gives_the_same_map(env, n, radius):
    G, ctx = env
    rng = np.random.default_rng(n)
    v, f = _soup(n, rng)
    tri = rng.integers(0, n, 700).astype(np.uint32)
    xyz = np.ascontiguousarray(v.reshape(-1, 3, 3)[tri].mean(1), np.float32)
    fix, ts = _look(60, rng), np.arange(60.0)
    got = []
    for kw in (dict(builder=G.GM_BUILD_PLOC, ploc_radius=radius), dict(builder=G.GM_BUILD_LBVH)):
        scene = G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)], **kw)
        nt, depth = G.gm_scene_info(scene)
        assert nt == n and math.ceil(math.log2(n)) <= depth <= min(64, n - 1)
        samples = G.gm_samples_from_points(scene, xyz, tri)
        got.append(_map(G, scene, samples, fix, ts))
        G.gm_samples_free(samples)
        G.gm_scene_free(scene)
    assert got[0][1]["visible"] == got[1][1]["visible"] > 0
    assert np.array_equal(got[0][0], got[1][0])


@pytest.mark.parametrize("nf,windows", [(1, 2), (33, 3), (2047, 5), (2048, 300), (2049, 5), (7000, 300)])
def test_sorted_windows_equal_single_intervals(env, nf, windows):
    G, ctx = env
    rng = np.random.default_rng(nf + windows)
    v, f = M.uv_sphere(12, 24, 1.0)
    scene = G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)])
    tri = rng.integers(0, len(f), 90).astype(np.uint32)
    xyz = np.ascontiguousarray(v[f[tri].astype(np.int64)].mean(1), np.float32)
    samples = G.gm_samples_from_points(scene, xyz, tri)
    fix, ts = _look(nf, rng), rng.uniform(-0.5, windows + 0.5, nf)      # in no order, some outside the interval
    out, st = _map(G, scene, samples, fix, ts, t_begin=0.0, t_end=float(windows), window_s=1.0)
    assert st["n_fixations_used"] == int(((ts >= 0) & (ts < windows)).sum())
    for w in sorted({0, windows // 2, windows - 1}):
        one, _ = _map(G, scene, samples, fix, ts, t_begin=float(w), t_end=float(w + 1))
        assert np.array_equal(out[w], one[0])
    G.gm_samples_free(samples)
    G.gm_scene_free(scene)


@pytest.mark.parametrize("copies,others", [(66, 0), (1100, 50), (4096, 0), (5000, 0), (5000, 300), (5200, 0), (20000, 100)])
def test_coincident_triangles_are_refused(env, copies, others):
    """Equal boxes merge one pair a round into a chain: a tree deeper than the traversal's 64 levels (from 4097
    levels on, deeper than its layout follows) is refused before it is laid out, and the next build works."""
    G, ctx = env
    rng = np.random.default_rng(copies + others)
    v, f = _soup(others + 1, rng)
    f = np.concatenate([f, np.repeat(f[:1], copies - 1, 0)])
    with pytest.raises(G.GazeMapError, match="deeper than 64 levels") as e:
        G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)])
    assert e.value.status == G.GM_ERR_UNSUPPORTED
    for n in (2, 40):      # a chain that is not too deep builds, and traces as the other builder's tree does
        f = np.repeat(f[:1], n, 0)
        xyz, tri = np.ascontiguousarray(v[:3].mean(0, keepdims=True)), np.zeros(1, np.uint32)
        fix, got = _look(60, rng), []
        for b in (G.GM_BUILD_PLOC, G.GM_BUILD_LBVH):
            scene = G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)], builder=b)
            samples = G.gm_samples_from_points(scene, xyz, tri)
            got.append(_map(G, scene, samples, fix, np.arange(60.0))[0])
            G.gm_samples_free(samples)
            G.gm_scene_free(scene)
        assert np.array_equal(got[0], got[1])
