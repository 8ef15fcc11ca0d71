"""The bounce wavefront of a histogram's initial stage is optional, so its scratch never takes the room of
anything that a call needs: under a budget of exactly what the scene, the views and the reuse scratch take,
every render and allocation succeeds and gives the bits of an unbounded context.  The wavefront's size is what
the first render of a view without reuse allocates."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes

pytestmark = pytest.mark.gpu

W, H, B = 24, 20, 40
BINS = (1.35, 1.024 / B, B)


def _context(sc, budget):
    from paper_2605_11536_gb300 import tof
    ctx = tof.tof_create(0, budget)
    sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
    tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
    return ctx, sid


def _frames(sc, ctx, sid, vid, n=3, first=0):
    import torch
    from paper_2605_11536_gb300 import tof
    out = torch.full((n, W * H * B), -1.0, device="cuda")
    for f in range(n):
        tof.tof_render_transient(ctx, sid, vid, sc.sensors[0], sc.emitters[0], BINS, sc.params, 3, first + f, out[f].data_ptr())
    tof.tof_sync(ctx)
    return out.cpu().numpy()


def _scene(temporal, nb):
    sc = scenes.confocal_nlos(W=W, H=H, frames=1, B=B, stacks=12, slices=12)
    sc.params.n_cand, sc.params.temporal, sc.params.n_spatial, sc.params.radius = 6, temporal, nb, 4
    return sc


def _wavefront_bytes():
    from paper_2605_11536_gb300 import tof
    sc = _scene(0, 0)
    ctx, sid = _context(sc, 0)
    try:
        vid = tof.tof_view_create(ctx, sid, W, H, B)
        before = tof.tof_device_bytes(ctx)
        _frames(sc, ctx, sid, vid, 1)
        return tof.tof_device_bytes(ctx) - before
    finally:
        tof.tof_destroy(ctx)


@pytest.mark.parametrize("temporal,nb", [(1, 2), (1, 0), (0, 3)])
def test_reuse_scratch_comes_before_the_wavefront(temporal, nb):
    from paper_2605_11536_gb300 import tof
    wave = _wavefront_bytes()
    assert wave > W * H * 6 * 100
    sc = _scene(temporal, nb)
    ctx, sid = _context(sc, 0)
    try:
        ref = _frames(sc, ctx, sid, tof.tof_view_create(ctx, sid, W, H, B))
        need = tof.tof_device_bytes(ctx) - wave
    finally:
        tof.tof_destroy(ctx)
    assert all(np.count_nonzero(r) > 20 for r in ref)
    for budget in (need, need + wave - 1, need + wave):
        ctx, sid = _context(sc, budget)
        try:
            np.testing.assert_array_equal(_frames(sc, ctx, sid, tof.tof_view_create(ctx, sid, W, H, B)), ref)
            assert tof.tof_device_bytes(ctx) == (budget if budget != need + wave - 1 else need)
        finally:
            tof.tof_destroy(ctx)
    ctx, sid = _context(sc, need - 1)   # and below what is needed it is refused, as before
    try:
        with pytest.raises(tof.TofError, match="budget"):
            _frames(sc, ctx, sid, tof.tof_view_create(ctx, sid, W, H, B))
    finally:
        tof.tof_destroy(ctx)


def test_a_later_view_takes_the_wavefronts_room():
    from paper_2605_11536_gb300 import tof
    wave = _wavefront_bytes()
    sc = _scene(0, 0)
    ctx, sid = _context(sc, 0)
    try:
        ref = _frames(sc, ctx, sid, tof.tof_view_create(ctx, sid, W, H, B))
        tof.tof_view_create(ctx, sid, W, H, B)
        need = tof.tof_device_bytes(ctx) - wave
    finally:
        tof.tof_destroy(ctx)
    ctx, sid = _context(sc, need)
    try:
        a = tof.tof_view_create(ctx, sid, W, H, B)
        np.testing.assert_array_equal(_frames(sc, ctx, sid, a, 1), ref[:1])
        assert tof.tof_device_bytes(ctx) < need   # with the wavefront: the second view is larger than it
        b = tof.tof_view_create(ctx, sid, W, H, B)
        np.testing.assert_array_equal(_frames(sc, ctx, sid, b), ref)
        np.testing.assert_array_equal(_frames(sc, ctx, sid, a, 2, 1), ref[1:])
        assert tof.tof_device_bytes(ctx) == need
    finally:
        tof.tof_destroy(ctx)


def test_changing_trees_and_depth_allocates_once():
    import torch
    from paper_2605_11536_gb300 import tof
    sc = _scene(0, 0)
    ctx, sid = _context(sc, 0)
    try:
        view, other = (tof.tof_view_create(ctx, sid, W, H, B) for _ in range(2))
        out = torch.full((2, W * H * B), -1.0, device="cuda")
        seen = []
        for f, (trees, depth) in enumerate([(8, 2), (4, 5), (8, 2), (4, 5), (1, 3), (8, 2)]):
            sc.params.n_cand, sc.params.depth = trees, depth
            tof.tof_render_transient(ctx, sid, view, sc.sensors[0], sc.emitters[0], BINS, sc.params, 3, f, out[0].data_ptr())
            seen.append(tof.tof_device_bytes(ctx))
            tof.tof_render_batch(ctx, [tof.job(sid, other, sc.sensors[0], sc.emitters[0], sc.params, 3, f, out[1].data_ptr(), bins=BINS)])
            tof.tof_sync(ctx)
            a = out.cpu().numpy()
            np.testing.assert_array_equal(a[0], a[1])   # in a batch: the single kernel
        assert seen[2:] == [seen[2]] * 4, seen
    finally:
        tof.tof_destroy(ctx)


@pytest.mark.parametrize("trees,depth,wave", [(1, 5, False), (3, 4, False), (4, 4, True), (8, 4, True)])
def test_few_trees_take_the_single_kernel(trees, depth, wave):
    import torch
    from paper_2605_11536_gb300 import tof
    sc = _scene(0, 0)
    sc.params.n_cand, sc.params.depth = trees, depth
    ctx, sid = _context(sc, 0)
    try:
        vid = tof.tof_view_create(ctx, sid, W, H, B)
        before = tof.tof_device_bytes(ctx)
        img = _frames(sc, ctx, sid, vid, 1)[0]
        assert (tof.tof_device_bytes(ctx) > before) == wave
        out = torch.full((W * H * B,), -1.0, device="cuda")   # a batch: always the single kernel
        tof.tof_render_batch(ctx, [tof.job(sid, vid, sc.sensors[0], sc.emitters[0], sc.params, 3, 0, out.data_ptr(), bins=BINS)])
        tof.tof_sync(ctx)
        np.testing.assert_array_equal(img, out.cpu().numpy())
        assert img.any()
    finally:
        tof.tof_destroy(ctx)
