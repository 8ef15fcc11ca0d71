"""A server's step builds the hierarchies of its frames' scenes beside one another: one scene, as many as there
are streams for it, more, and two streams of one scene (never in one step).  Every frame equals the direct
render of its scene bit for bit."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes

pytestmark = pytest.mark.gpu
NF = 3


@pytest.mark.parametrize("n,shared", [(1, 0), (2, 0), (4, 0), (7, 0), (3, 2)])
def test_scenes_built_beside_one_another_render_as_alone(n, shared):
    import torch
    from paper_2605_11536_gb300 import tof
    scs = [scenes.heightfield_spheres(W=40 + 8 * i, H=32, frames=NF, nx=30 + 25 * i, ny=20 + 7 * i, n_spheres=3 + i) for i in range(n)]
    of = list(range(n)) + [0] * shared   # scene of each stream
    imgs = []
    for served in (0, 1):
        ctx = tof.tof_create(0)
        try:
            sids = []
            for sc in scs:
                sc.params.radius, sc.params.temporal = 8, 1
                sids.append(tof.tof_scene_upload(ctx, sc.verts, sc.tris, sc.tri_object, sc.materials, sc.object_material))
                tof.tof_bvh_build(ctx, sids[-1], sc.xforms[0].reshape(-1))
            out = [[torch.full((sc.sensors[0]["W"] * 32,), -1.0, device="cuda") for _ in range(NF)] for sc in (scs[k] for k in of)]
            if served:
                srv = tof.tof_server_create(ctx, 0)
                streams = [tof.tof_server_open_stream(srv, sids[k], scs[k].sensors[0]["W"], 32, 0) for k in of]
                tickets = []
                for f in range(NF):
                    for i, k in enumerate(of):
                        sc = scs[k]
                        j = tof.job(sids[k], 0, sc.sensors[f], sc.emitters[f], sc.params, 5 + i, f, out[i][f].data_ptr(), gate=sc.gates[f])
                        tickets.append(tof.tof_server_submit(srv, streams[i], j, sc.xforms[f].reshape(-1)))
                    while tickets:
                        tof.tof_server_step(srv)
                        tickets = [t for t in tickets if tof.tof_server_poll(srv, t)[0] != 2]
                tof.tof_server_destroy(srv)
            else:
                views = [tof.tof_view_create(ctx, sids[k], scs[k].sensors[0]["W"], 32, 0) for k in of]
                for f in range(NF):
                    for i, k in enumerate(of):
                        sc = scs[k]
                        tof.tof_bvh_build(ctx, sids[k], sc.xforms[f].reshape(-1))
                        tof.tof_render_gated(ctx, sids[k], views[i], sc.sensors[f], sc.emitters[f], sc.gates[f], sc.params, 5 + i, f,
                                             out[i][f].data_ptr())
                tof.tof_sync(ctx)
            torch.cuda.synchronize()
            imgs.append([b.cpu().numpy() for o in out for b in o])
        finally:
            tof.tof_destroy(ctx)
    for a, b in zip(*imgs):
        np.testing.assert_array_equal(a, b)
    assert sum(np.count_nonzero(a) for a in imgs[0]) > 20
