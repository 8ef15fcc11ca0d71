"""A batch's persistent reuse stages give every instance a share of the grid's warps that starts where the
last instance's ended: instances of one pixel and without any task, shares that wrap around the grid, one
instance longer than the grid's lanes, two to nine slots.  Every view equals its direct render bit for bit."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,nb,flags", [
    ([(1, 1), (33, 7), (1, 1), (64, 64), (5, 40), (31, 1), (2, 2), (17, 19), (48, 3)], 3, 0),
    ([(96, 96)] * 20 + [(1, 1), (3, 50)], 8, 0),
    ([(640, 480), (16, 16), (1, 1), (64, 64), (31, 33), (128, 8)], 1, scenes.FLAG_DIRECT),
    ([(50, 20)] * 6 + [(7, 7)], 4, scenes.FLAG_PAIRWISE_MIS),
])
def test_shares_of_a_batch_equal_direct_renders(sizes, nb, flags):
    import torch
    from paper_2605_11536_gb300 import tof
    sc = scenes.box_materials(W=64, H=64, frames=1)
    p = sc.params
    p.n_spatial, p.temporal, p.flags = nb, 1, flags
    ctx = tof.tof_create(0)
    try:
        sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
        tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
        views = [[tof.tof_view_create(ctx, sid, w, h, 0) for w, h in sizes] for _ in range(2)]
        out = [[torch.full((w * h,), -1.0, device="cuda") for w, h in sizes] for _ in range(2)]
        emitter = sc.emitters[0]
        for f in range(2):
            jobs = []
            for i, (w, h) in enumerate(sizes):
                sensor = dict(sc.sensors[0], W=w, H=h)
                # every third view's gate lies beyond every path: its stages have no task
                gate = (1000.0, sc.gates[0][1]) if i % 3 == 2 else sc.gates[0]
                tof.tof_render_gated(ctx, sid, views[0][i], sensor, emitter, gate, p, 3 + i, f, out[0][i].data_ptr())
                jobs.append(tof.job(sid, views[1][i], sensor, emitter, p, 3 + i, f, out[1][i].data_ptr(), gate=gate))
            tof.tof_render_batch(ctx, jobs)
            tof.tof_sync(ctx)
            for i in range(len(sizes)):
                a, b = out[0][i].cpu().numpy(), out[1][i].cpu().numpy()
                np.testing.assert_array_equal(a, b)
                if i % 3 == 2:
                    assert not a.any()
        assert max(np.count_nonzero(x.cpu().numpy()) for x in out[0]) > 20
    finally:
        tof.tof_destroy(ctx)
