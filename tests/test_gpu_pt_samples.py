"""Plain path tracing at sample counts that do not divide a block, in images large enough that a block takes
several pixels over several rounds (pixels whose samples begin in one round and end in another), against the
FP64 oracle at the parity bar."""
import numpy as np
import pytest

from paper_2605_11536_gb300 import scenes
from tests.harness import PARITY_FRAC, PARITY_RELMSE, compare, gpu_pt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,spp,B", [(128, 128, 65, 0), (130, 126, 33, 0), (96, 130, 129, 0), (101, 127, 43, 9), (64, 41, 64, 0),
                                       (128, 96, 100, 3)])
def test_samples_that_do_not_divide_a_block(W, H, spp, B):
    import oracle as O
    sc = scenes.box_icosphere(W=W, H=H)
    sc.gates, sc.bins = [(5.0, 0.5)], (4.5, 0.25, B)
    sc.params.depth = 3
    g = gpu_pt(sc, 0, spp, seed=3, B=B)
    o = O.render_pt(O.Geom(sc, 0), sc, 0, spp=spp, seed=3, **({"B": B} if B else {}))
    frac, relmse, _ = compare(g, o)
    assert frac >= PARITY_FRAC and relmse <= PARITY_RELMSE, (frac, relmse)
    assert np.count_nonzero(g) > W * H // 4
