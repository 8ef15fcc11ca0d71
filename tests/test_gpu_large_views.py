"""Gated views of more than 16M pixels x trees, whose initial stage has no wavefront scratch and a thread per pixel:
the oracle at the parity bar in a region, and a batch of the same view (beside a small one) bit for bit."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes
from tests.harness import PARITY_FRAC, PARITY_RELMSE, compare, oracle_render

pytestmark = pytest.mark.gpu


def test_a_view_beyond_the_wavefronts_limit():
    import torch
    from paper_2605_11536_gb300 import tof
    W, H = 1040, 1017
    sc = scenes.box_icosphere(W=W, H=H)
    sc.gates = [(5.0, 0.5)]
    p = sc.params
    p.n_cand, p.depth, p.n_spatial, p.temporal = 16, 3, 0, 0
    assert W * H * p.n_cand > 16 * 1024 * 1024
    ctx = tof.tof_create(0)
    try:
        sid = tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material)
        tof.tof_bvh_build(ctx, sid, sc.xforms[0].reshape(-1))
        views = [tof.tof_view_create(ctx, sid, w, h, 0) for w, h in ((W, H), (W, H), (32, 20), (32, 20))]
        out = [torch.full((n,), -1.0, device="cuda") for n in (W * H, W * H, 640, 640)]
        small = dict(sc.sensors[0], W=32, H=20)
        tof.tof_render_gated(ctx, sid, views[0], sc.sensors[0], sc.emitters[0], sc.gates[0], p, 3, 0, out[0].data_ptr())
        tof.tof_render_gated(ctx, sid, views[2], small, sc.emitters[0], sc.gates[0], p, 3, 0, out[2].data_ptr())
        tof.tof_render_batch(ctx, [tof.job(sid, views[k], s, sc.emitters[0], p, 3, 0, out[k].data_ptr(), gate=sc.gates[0])
                                   for k, s in ((1, sc.sensors[0]), (3, small))])
        tof.tof_sync(ctx)
        img = [o.cpu().numpy() for o in out]
    finally:
        tof.tof_destroy(ctx)
    np.testing.assert_array_equal(img[0], img[1])
    np.testing.assert_array_equal(img[2], img[3])
    roi = (500, 480, 564, 544)
    ref, ok, _, _ = oracle_render(sc, [0], seed=3, roi=roi)
    sel = (slice(roi[1], roi[3]), slice(roi[0], roi[2]))
    frac, relmse, _ = compare(img[0].reshape(H, W)[sel], ref[0][sel])
    assert np.count_nonzero(ref[0][sel]) > 400   # 411: the gate takes a corner of the region
    assert frac >= PARITY_FRAC and relmse <= PARITY_RELMSE, (frac, relmse)
