"""The hierarchy's treelets and the levels above them: plain path tracing (first hits, bounces and light
segments) of triangle soups against the FP64 oracle, which has its own hierarchy, at triangle counts
around a treelet, a warp and a power of two, and with coincident triangles (splits that cannot tell them
apart); and a refit of the topology against a full build of the same transforms, whose images are equal
bit for bit (a hit does not depend on the hierarchy), also with more ranges than the top kernel takes."""
import math

import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes
from tests.harness import PARITY_FRAC, PARITY_RELMSE, compare, gpu_pt

pytestmark = pytest.mark.gpu


def _soup(n, W, H, seed=0, coincident=0, size=0.25, frames=1, objects=1):
    rng = np.random.default_rng(seed)
    c = rng.uniform([-1.2, -0.9, -3.6], [1.2, 0.9, -2.4], size=(n, 1, 3))
    v = c + rng.uniform(-size, size, size=(n, 3, 3))
    if coincident:
        v[:coincident] = v[0]
    if n < 8:
        v[0] = [[-4, -3, -4.0], [4, -3, -4.2], [0, 5, -3.8]]
    sc = scenes.lambert_plane(W=W, H=H)
    sc.verts, sc.tris = v.reshape(-1, 3), np.arange(3 * n, dtype=np.uint32).reshape(n, 3)
    sc.tri_object = (np.arange(n, dtype=np.uint32) * objects // n).astype(np.uint32)
    sc.object_material = np.zeros(objects, dtype=np.uint32)
    sc.xforms = np.tile(np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], dtype=np.float64), (frames, objects, 1))
    for f in range(frames):
        for o in range(1, objects):
            a = 0.1 * f * o
            sc.xforms[f, o] = [math.cos(a), -math.sin(a), 0, 0.02 * f, math.sin(a), math.cos(a), 0, 0, 0, 0, 1, -0.03 * f]
    sc.sensors, sc.emitters, sc.gates = sc.sensors * frames, sc.emitters * frames, [(0.0, 1.0e3)] * frames
    sc.params.depth, sc.params.flags = 3, scenes.FLAG_DIRECT
    return sc


@pytest.mark.parametrize("n,coincident", [(1, 0), (2, 0), (3, 0), (33, 0), (511, 0), (512, 0), (513, 0), (1024, 0), (2500, 0), (700, 600)])
def test_soup_matches_the_oracle(n, coincident):
    import oracle as O
    sc = _soup(n, 64, 48, seed=n, coincident=coincident)
    g = gpu_pt(sc, 0, 4, seed=5)
    o = O.render_pt(O.Geom(sc, 0), sc, 0, spp=4, seed=5)
    frac, relmse, _ = compare(g, o)
    assert np.count_nonzero(o) > 100
    assert frac >= PARITY_FRAC and relmse <= PARITY_RELMSE, (frac, relmse)


@pytest.mark.parametrize("n,size", [(3, 0.25), (400, 0.25), (700, 0.25), (6000, 0.1), (900_000, 0.006)])   # the last: over 1024 ranges
def test_refit_of_the_topology_equals_a_full_build(n, size):
    import torch
    from paper_2605_11536_gb300 import tof
    sc = _soup(n, 64, 48, seed=n, size=size, frames=3, objects=3)
    imgs = []
    for refit in (0, 1):
        ctx = tof.tof_create(0)
        try:
            sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
            out = torch.zeros(64 * 48, device="cuda")
            for f in range(3):
                tof.tof_bvh_build(ctx, sid, sc.xforms[f].reshape(-1), refit_only=refit)
            tof.tof_render_pt(ctx, sid, sc.sensors[2], sc.emitters[2], sc.gates[2], None, sc.params, 5, 0, 4, out.data_ptr())
            tof.tof_sync(ctx)
            imgs.append(out.cpu().numpy().copy())
        finally:
            tof.tof_destroy(ctx)
    np.testing.assert_array_equal(imgs[0], imgs[1])
    assert np.count_nonzero(imgs[0]) > 100
