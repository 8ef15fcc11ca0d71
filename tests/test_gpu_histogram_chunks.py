"""A histogram's reuse passes take as many pixels at a time as their occupied bins can need, bounded from the
candidates and the passes of the frames so far; a batch still divides by all bins.  Both equal each other bit
for bit over a history that fills up: several chunks, one, bins that do not divide a word, bin reuse, the
ellipsoidal connection, a history that is forgotten midway, and renders in a batch between direct ones."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,B,trees,nb,flags", [
    (96, 64, 1024, 8, 3, 0), (33, 31, 5000, 2, 8, scenes.FLAG_BIN_REUSE), (130, 40, 999, 4, 2, scenes.FLAG_ELLIPSOID),
    (64, 70, 1000, 8, 0, scenes.FLAG_DIRECT), (20, 20, 64, 3, 1, 0)])
def test_chunks_by_occupied_bins_equal_chunks_by_all_bins(W, H, B, trees, nb, flags):
    import torch
    from paper_2605_11536_gb300 import tof
    sc = scenes.confocal_nlos(W=W, H=H, frames=4, B=B, stacks=24, slices=24)
    p = sc.params
    p.n_cand, p.n_spatial, p.temporal, p.flags = trees, nb, 1, flags
    if flags & scenes.FLAG_DIRECT or flags & scenes.FLAG_ELLIPSOID:
        p.n_cand = min(trees, 4)
    bins = (1.35, 1.024 / B, B)
    ctx = tof.tof_create(0)
    try:
        sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
        tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
        out = torch.full((2, W * H * B), -1.0, device="cuda")
        views = [tof.tof_view_create(ctx, sid, W, H, B) for _ in range(2)]
        for f in range(6):
            k = f % 4
            if f == 4:
                for v in views:
                    tof.tof_reservoirs_reset(ctx, v)

            def batch(i):
                tof.tof_render_batch(ctx, [tof.job(sid, views[i], sc.sensors[k], sc.emitters[k], p, 3, f, out[i].data_ptr(), bins=bins)])
            if f == 2:
                batch(0)   # between direct renders of the same view
            else:
                tof.tof_render_transient(ctx, sid, views[0], sc.sensors[k], sc.emitters[k], bins, p, 3, f, out[0].data_ptr())
            batch(1)
            tof.tof_sync(ctx)
            a = out.cpu().numpy()
            np.testing.assert_array_equal(a[0], a[1])
        assert np.count_nonzero(a[0]) >= 20
    finally:
        tof.tof_destroy(ctx)
