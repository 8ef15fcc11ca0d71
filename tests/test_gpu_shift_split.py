"""The shift kernels run records that reconnect at their second vertex in their loop and put the
others (glossy and mirror prefixes, replayed) off to the warp's end.  Every task is shifted once
however it is split: the numbers of forward shifts and of Newton solves of a box with glossy and mirror
walls, at sizes with a partial warp, a few put-off tasks a warp and lists longer than a warp, are the
oracle's, up to branch flips (the bar of the other shift-count test)."""
import pytest

from paper_2605_11536_gb300 import scenes
from tests.harness import gpu_render, oracle_render

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(5, 3), (19, 13), (64, 48)])
def test_every_shift_runs_once(W, H):
    sc = scenes.box_materials(W=W, H=H, frames=3, moving=True)
    sc.gates = [(6.0, 1.0)] * 3
    p = sc.params
    p.n_spatial, p.radius, p.temporal, p.depth = 5, 6, 1, 5
    _, g = gpu_render(sc, [0, 1, 2], collect_stats=True)
    o = oracle_render(sc, [0, 1, 2])[2]
    for k in ("shift_calls", "newton_calls", "inv_calls"):
        if k in o:
            assert abs(g[k] - o[k]) <= 0.02 * o[k] + 2, (k, g[k], o[k])
    if W * H > 1000:
        assert g["shift_calls"] > 1000
