"""Path trees in lanes (the allocation-free gated form), the bounce wavefront for histograms and plain path
tracing with a thread per sample: each draws the numbers of the form it replaces in the same order, so it
equals the other form of the same render bit for bit (a histogram in a batch keeps the single kernel), or
the FP64 oracle at the parity bar where there is no other form.  Tree and sample counts that do not
divide a block, one, and more than a block takes at once; ragged views; bins that share words."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes
from tests.harness import PARITY_FRAC, PARITY_RELMSE, compare, gpu_pt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,trees,depth,flags", [(1, 1, 1, 3, 0), (13, 9, 3, 5, scenes.FLAG_DIRECT), (31, 5, 7, 2, 0), (9, 17, 64, 3, 0),
                                                   (64, 50, 5, 4, 0)])
def test_trees_in_lanes_equal_the_wavefront(W, H, trees, depth, flags):
    import torch
    from paper_2605_11536_gb300 import tof
    sc = scenes.box_materials(W=W, H=H, frames=1)
    p = sc.params
    p.n_cand, p.depth, p.n_spatial, p.temporal, p.flags = trees, depth, 2, 1, flags
    ctx = tof.tof_create(0)
    try:
        sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
        tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
        out = torch.full((2, W * H), -1.0, device="cuda")
        views = [tof.tof_view_create(ctx, sid, W, H, 0) for _ in range(2)]
        for f in range(2):
            for k, call in enumerate((tof.tof_render_gated, tof.tof_render_gated_noalloc)):
                call(ctx, sid, views[k], sc.sensors[0], sc.emitters[0], sc.gates[0], p, 3, f, out[k].data_ptr())
            tof.tof_sync(ctx)
            a = out.cpu().numpy()
            np.testing.assert_array_equal(a[0], a[1])
        if W * H * trees > 1000:
            assert np.count_nonzero(a[0]) > 20
    finally:
        tof.tof_destroy(ctx)


@pytest.mark.parametrize("W,H,B,trees,flags", [(5, 3, 1, 2, 0), (16, 11, 33, 8, scenes.FLAG_DIRECT), (24, 24, 700, 5, 0)])
def test_histogram_wavefront_equals_the_single_kernel(W, H, B, trees, flags):
    import torch
    from paper_2605_11536_gb300 import tof
    sc = scenes.confocal_nlos(W=W, H=H, frames=2, B=B, stacks=24, slices=24)
    p = sc.params
    p.n_cand, p.flags = trees, flags
    bins = (1.35, 1.024 / B, B)
    ctx = tof.tof_create(0)
    try:
        sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
        tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
        out = torch.full((2, W * H * B), -1.0, device="cuda")
        views = [tof.tof_view_create(ctx, sid, W, H, B) for _ in range(2)]
        for f in range(2):
            tof.tof_render_transient(ctx, sid, views[0], sc.sensors[f], sc.emitters[f], bins, p, 3, f, out[0].data_ptr())
            tof.tof_render_batch(ctx, [tof.job(sid, views[1], sc.sensors[f], sc.emitters[f], p, 3, f, out[1].data_ptr(), bins=bins)])
            tof.tof_sync(ctx)
            a = out.cpu().numpy()
            np.testing.assert_array_equal(a[0], a[1])
        assert np.count_nonzero(a[0]) >= min(W * H // 4, 20)
    finally:
        tof.tof_destroy(ctx)


def test_histogram_without_room_for_the_wavefront_renders_all_the_same():
    import torch
    from paper_2605_11536_gb300 import tof
    W = H = 16
    sc = scenes.confocal_nlos(W=W, H=H, frames=1, B=8, stacks=12, slices=12)
    sc.params.temporal, sc.params.n_spatial = 0, 0
    imgs = []
    for budget in (0, None):
        ctx = tof.tof_create(0, budget or 0)
        if budget is None:   # exactly what the scene and the view take
            tof.tof_destroy(ctx)
            ctx = tof.tof_create(0, need)
        try:
            sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
            tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
            vid = tof.tof_view_create(ctx, sid, W, H, 8)
            need = tof.tof_device_bytes(ctx)
            out = torch.full((W * H * 8,), -1.0, device="cuda")
            for f in range(2):
                tof.tof_render_transient(ctx, sid, vid, sc.sensors[0], sc.emitters[0], (1.35, 0.128, 8), sc.params, 3, f, out.data_ptr())
            tof.tof_sync(ctx)
            if budget is None:
                assert tof.tof_device_bytes(ctx) == need
            imgs.append(out.cpu().numpy().copy())
        finally:
            tof.tof_destroy(ctx)
    np.testing.assert_array_equal(imgs[0], imgs[1])
    assert np.count_nonzero(imgs[0]) > 20


@pytest.mark.parametrize("W,H,spp,B", [(1, 1, 1, 0), (33, 7, 5, 0), (12, 5, 300, 0), (16, 9, 24, 40)])
def test_path_tracing_with_a_thread_per_sample(W, H, spp, B):
    import oracle as O
    sc = scenes.box_icosphere(W=W, H=H)
    sc.gates, sc.bins = [(5.0, 0.5)], (4.5, 0.05, B)
    sc.params.depth = 4
    g = gpu_pt(sc, 0, spp, seed=3, B=B)
    o = O.render_pt(O.Geom(sc, 0), sc, 0, spp=spp, seed=3, **({"B": B} if B else {}))
    frac, relmse, _ = compare(g, o)
    # a value that one sample moves into the next bin or across the gate takes one or two of them
    assert frac >= min(PARITY_FRAC, 1.0 - 2.0 / g.size) and relmse <= PARITY_RELMSE, (frac, relmse)
