"""Records that replay past their second vertex (behind mirrors and glossy walls), which the shift kernels put off
to the warp's end: in a room whose visible wall is a mirror most records are such, so a put-off task that
did not run would show, a forward one as a lost sample and an inverse one as a lost term of the MIS weight.  Images
against the FP64 oracle at the parity bar, and the oracle's numbers of forward shifts and Newton solves within
the branch flips of the other shift-count test; temporal and spatial reuse, sizes with partial warps."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes
from tests.harness import PARITY_FRAC, PARITY_RELMSE, compare, gpu_render, oracle_render


def _scene(W, H, temporal):
    sc = scenes.box_materials(W=W, H=H, frames=2, sphere_alpha=0.5)
    om = sc.object_material.copy()
    om[0], om[1] = 1, 0   # the wall that the camera sees is a mirror, the one behind it is rough
    sc.object_material = om
    sc.gates = [(10.0, 3.0)] * 2
    p = sc.params
    p.n_spatial, p.radius, p.temporal, p.depth = 3, 6, temporal, 5
    return sc


def _most_records_replay(sc):
    import oracle as O
    s = sc.sensors[0]
    W, H = int(s["W"]), int(s["H"])
    v = O.View(W, H, 0)
    g = O.Geom(sc, 0)
    O.render_frame(v, g, sc, 0)
    r = [v.reservoir(p) for p in range(W * H)]
    r = [x["r"] for x in r if x["valid"]]
    return len(r), sum(x > 2 for x in r) / max(1, len(r))


def test_most_records_of_the_scene_replay():
    n, share = _most_records_replay(_scene(32, 24, 0))
    assert n > 300 and share > 0.6, (n, share)


@pytest.mark.gpu
@pytest.mark.parametrize("W,H,temporal", [(61, 43, 0), (64, 48, 1)])
def test_replayed_shifts_match_the_oracle(W, H, temporal):
    sc = _scene(W, H, temporal)
    imgs, g = gpu_render(sc, [0, 1], collect_stats=True)
    refs, _, o, _ = oracle_render(sc, [0, 1])
    for k in ("shift_calls", "newton_calls"):
        assert o[k] > 2000 and abs(g[k] - o[k]) <= 0.02 * o[k] + 2, (k, g[k], o[k])
    assert g["inv_calls"] > o["shift_ok"]   # every shifted candidate is shifted into the other domains
    for img, ref in zip(imgs, refs):
        frac, relmse, _ = compare(img, ref)
        assert np.count_nonzero(ref) > W * H // 4
        assert frac >= PARITY_FRAC and relmse <= PARITY_RELMSE, (frac, relmse)
