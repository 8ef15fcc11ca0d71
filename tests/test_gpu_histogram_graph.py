"""A histogram frame recorded into a graph holds the view's wavefront scratch by address: later renders of the
view with more path trees or longer paths leave that scratch where it is (they take the single kernel), and a
replay gives the recorded frame."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recorded_with_scratch", [True, False])
def test_a_recorded_frame_keeps_its_scratch(recorded_with_scratch):
    import torch
    from paper_2605_11536_gb300 import tof
    W, H, B = 24, 20, 40
    sc = scenes.confocal_nlos(W=W, H=H, frames=1, B=B, stacks=12, slices=12)
    bins = (1.35, 1.024 / B, B)
    p = sc.params
    p.temporal, p.n_spatial, p.radius = 0, 2, 4
    ctx = tof.tof_create(0)
    try:
        sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
        tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
        vid = tof.tof_view_create(ctx, sid, W, H, B)

        def render(trees, depth, frame, out, stream=0):
            p.n_cand, p.depth = trees, depth
            tof.tof_render_transient(ctx, sid, vid, sc.sensors[0], sc.emitters[0], bins, p, 3, frame, out.data_ptr(), stream)

        ref, out, rec = (torch.full((W * H * B,), -1.0, device="cuda") for _ in range(3))
        if not recorded_with_scratch:   # the reuse scratch alone, by the form that takes no other
            p.n_cand, p.depth = 4, 3
            tof.tof_render_batch(ctx, [tof.job(sid, vid, sc.sensors[0], sc.emitters[0], p, 3, 5, ref.data_ptr(), bins=bins)])
        else:
            render(4, 3, 5, ref)
        tof.tof_sync(ctx)
        held = tof.tof_device_bytes(ctx)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            render(4, 3, 5, rec, torch.cuda.current_stream().cuda_stream)
        assert tof.tof_device_bytes(ctx) == held
        seen = []
        for trees, depth in ((8, 4), (5, 4), (8, 2), (4, 3)):
            render(trees, depth, 5, out)
            tof.tof_sync(ctx)
            seen.append(tof.tof_device_bytes(ctx))
            assert np.count_nonzero(out.cpu().numpy()) > 20
        if recorded_with_scratch:
            assert seen == [held] * 4
        else:   # taken after the recording, by the first of them
            assert seen[0] > held and seen == [seen[0]] * 4
        for _ in range(2):
            rec.fill_(-1.0)
            graph.replay()
            torch.cuda.synchronize()
            np.testing.assert_array_equal(rec.cpu().numpy(), ref.cpu().numpy())
        np.testing.assert_array_equal(out.cpu().numpy(), ref.cpu().numpy())   # (4, 3) again
    finally:
        torch.cuda.synchronize()
        tof.tof_destroy(ctx)
