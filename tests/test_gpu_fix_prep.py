"""Lists of up to 2048 fixations and windows are prepared by one block, longer ones by separate kernels:
the same fixations through both (one list is made longer by fixations outside the interval) give the same maps, maxima and counts bit for bit."""
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


@pytest.mark.parametrize("nf,windows,into", [
    (1, 1, False), (31, 1, False), (1024, 2, False), (1025, 255, False), (2047, 256, False), (2048, 300, False),
    (700, 2048, False), (1, 1, True), (1025, 3, True), (2048, 2, True)])
def test_one_block_preparation_equals_the_kernels(env, nf, windows, into):
    G, ctx = env
    v, f = M.uv_sphere(12, 24, 1.0)
    scene = G.gm_build_scene(ctx, [(v, f, np.eye(4), 0)], dynamic=into)
    samples = G.gm_sample_surface(scene, [40.0], 7)
    ns = G.gm_samples_info(samples)

    def run(extra):
        r = np.random.default_rng(nf)
        n = nf + extra
        eye = r.normal(size=(nf, 3))
        eye *= 2.5 / np.maximum(np.linalg.norm(eye, axis=1, keepdims=True), 1e-9)
        gaze = 0.3 * r.normal(size=(nf, 3)) - eye
        dur = r.uniform(0.1, 0.6, nf)
        ts = np.concatenate([r.uniform(0.0, windows, nf), np.full(extra, windows + 1.0)])
        pad = np.ones((extra, 3))
        # the ignored ones stand between the others
        at = np.arange(n) if extra == 0 else np.argsort(np.concatenate([np.arange(nf), r.uniform(0, nf, extra)]), kind="stable")
        fix = [np.ascontiguousarray(np.concatenate([eye, pad])[at], np.float32),
               np.ascontiguousarray(np.concatenate([gaze, pad])[at], np.float32),
               np.concatenate([dur, np.ones(extra)])[at].astype(np.float32), np.ascontiguousarray(ts[at])]
        prm = G.make_params(math.radians(6.0), t_begin=0.0, t_end=float(windows), window_s=1.0)
        if into:
            m = G.gm_accumulate_dynamic(scene, samples, *fix, prm, np.broadcast_to(np.eye(4), (windows, 1, 4, 4)))
        else:
            m = G.gm_accumulate_fixations(scene, samples, *fix, prm)
        W, _, st, _ = G.gm_map_info(m)
        maps = np.empty((W, ns), np.float32)
        top = [G.gm_map_copy(m, w, maps[w]) for w in range(W)]
        G.gm_map_free(m)
        return maps, top, {k: st[k] for k in ("in_cone", "visible")}

    one, many = run(0), run(2049 - nf)
    G.gm_samples_free(samples)
    G.gm_scene_free(scene)
    assert one[1] == many[1] and one[2] == many[2]
    assert np.array_equal(one[0], many[0])
    if nf > 30:
        assert one[2]["visible"] > 0
