"""Full builds at the triangle counts where their forms change: one block for the whole scene, the sort whose
blocks add up the histograms, the one with scanned rows, the separate launches, and the levels above more than
1024 ranges in one block or over the GPU.  Path tracing against the FP64 oracle at small counts; at large
ones the build of the last transforms against the build of the first refitted to them (the Morton order and
the hierarchy are others, the images equal bit for bit)."""
import numpy as np
import pytest

from tests.harness import PARITY_FRAC, PARITY_RELMSE, compare, gpu_pt
from tests.test_gpu_treelets import _soup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,coincident", [(31, 0), (32, 0), (257, 0), (512, 500), (900, 0), (1023, 0), (1024, 1000), (1025, 0), (1025, 1025), (3000, 2000)])
def test_build_matches_the_oracle(n, coincident):
    import oracle as O
    sc = _soup(n, 64, 48, seed=n + 1, coincident=coincident)
    if coincident == n:   # one triangle many times: make it one that fills the view
        sc.verts[:] = np.tile(np.array([[-4, -3, -4.0], [4, -3, -4.2], [0, 5, -3.8]]), (n, 1))
    g = gpu_pt(sc, 0, 4, seed=5)
    o = O.render_pt(O.Geom(sc, 0), sc, 0, spp=4, seed=5)
    frac, relmse, _ = compare(g, o)
    assert np.count_nonzero(o) > 10
    assert frac >= PARITY_FRAC and relmse <= PARITY_RELMSE, (frac, relmse)


@pytest.mark.parametrize("n,size", [(512, 0.25), (1024, 0.25), (1025, 0.25), (56_320, 0.03), (56_321, 0.03), (262_144, 0.012), (262_145, 0.012),
                                    (307_200, 0.012), (307_201, 0.012), (700_000, 0.008)])
def test_a_refit_equals_a_full_build(n, size):
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
