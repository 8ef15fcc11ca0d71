"""Queued rays (trace_queue: the visibility segments and the bounce wavefront's closest hits) against
the same rays traced in place: a direct render queues every light segment and bounce ray of its
initial stage, the allocation-free form traces them inside its kernel, and both trace the same rays,
so the images are equal bit for bit.  The sizes bring fewer rays than the grid has warps (a warp then
takes only its share), a remainder, and more; scenes of one and two triangles have no hierarchy or a
single node."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes

pytestmark = pytest.mark.gpu


def _frames(sc, W, H, entry, frames=2):
    import torch
    from paper_2605_11536_gb300 import tof
    ctx = tof.tof_create(0)
    try:
        sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
        vid = tof.tof_view_create(ctx, sid, W, H, 0)
        tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
        out = torch.full((W * H,), -1.0, device="cuda")
        imgs = []
        for f in range(frames):
            getattr(tof, entry)(ctx, sid, vid, sc.sensors[0], sc.emitters[0], sc.gates[0], sc.params, 5, f, out.data_ptr())
            tof.tof_sync(ctx)
            imgs.append(out.cpu().numpy().copy())
        return imgs
    finally:
        tof.tof_destroy(ctx)


@pytest.mark.parametrize("W,H", [(1, 1), (7, 5), (33, 3), (129, 1), (128, 128)])
def test_queued_rays_equal_rays_traced_in_place(W, H):
    sc = scenes.box_icosphere(W=W, H=H)
    sc.gates = [(5.0, 0.5)]
    sc.params.n_spatial, sc.params.radius, sc.params.temporal, sc.params.n_cand = 3, 4, 1, 5
    a, b = _frames(sc, W, H, "tof_render_gated"), _frames(sc, W, H, "tof_render_gated_noalloc")
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
    if W * H > 1000:
        assert np.count_nonzero(a[0]) > 100


@pytest.mark.parametrize("nt", [1, 2])
def test_queued_rays_of_one_and_two_triangles(nt):
    sc = scenes.lambert_plane(W=24, H=9)
    sc.tris, sc.tri_object = sc.tris[:nt], sc.tri_object[:nt]
    a, b = _frames(sc, 24, 9, "tof_render_gated"), _frames(sc, 24, 9, "tof_render_gated_noalloc")
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
    assert np.count_nonzero(a[0]) > 10
