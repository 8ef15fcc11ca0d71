"""Path trees in lanes at tree counts that do not divide a block, in launches large enough that a block takes
several rounds and a pixel's trees reach over two of them: the allocation-free form and a batch equal the bounce
wavefront of a direct render bit for bit."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,trees,depth,flags", [(128, 128, 43, 3, 0), (121, 101, 21, 5, scenes.FLAG_DIRECT), (128, 97, 33, 2, 0),
                                                   (100, 127, 50, 3, 0), (127, 128, 7, 4, 0)])
def test_rounds_of_trees_equal_the_wavefront(W, H, trees, depth, flags):
    import torch
    from paper_2605_11536_gb300 import tof
    n = 5
    sc = scenes.box_materials(W=W, H=H, frames=1)
    p = sc.params
    p.n_cand, p.depth, p.n_spatial, p.temporal, p.flags = trees, depth, 1, 1, flags
    ctx = tof.tof_create(0)
    try:
        sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
        tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
        out = torch.full((2 + n, W * H), -1.0, device="cuda")
        views = [tof.tof_view_create(ctx, sid, W, H, 0) for _ in range(2 + n)]
        for f in range(2):
            for k, call in enumerate((tof.tof_render_gated, tof.tof_render_gated_noalloc)):
                call(ctx, sid, views[k], sc.sensors[0], sc.emitters[0], sc.gates[0], p, 3, f, out[k].data_ptr())
            tof.tof_render_batch(ctx, [tof.job(sid, views[2 + i], sc.sensors[0], sc.emitters[0], p, 3, f, out[2 + i].data_ptr(),
                                               gate=sc.gates[0]) for i in range(n)])
            tof.tof_sync(ctx)
            a = out.cpu().numpy()
            for k in range(1, 2 + n):
                np.testing.assert_array_equal(a[0], a[k])
        assert np.count_nonzero(a[0]) > W * H // 20
    finally:
        tof.tof_destroy(ctx)
