"""A batch solves with the walls it was created with, whatever is set on its
views later: the tables that its launches name stay allocated."""
import numpy as np
import pytest

from paper_1801_04577_gb300 import clbm
from paper_1801_04577_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_walls_set_on_views_do_not_reach_the_batch(precision):
    torch = pytest.importorskip("torch")
    # resident boxes and obstacles, tiles without and with a mask (FP64: all tiles)
    ws = [I.natural_convection_cavity(24, 1e4), I.obstacle_cavities(1, 32)[0], I.natural_convection_cavity(300, 1e4),
          I.obstacle_channel(500, 120)]
    plain, changed = clbm.Batch(ws, precision), clbm.Batch(ws, precision)
    plain.solve(0.0, 20, 10)
    changed.solve(0.0, 20, 10)
    keep = []
    for i, w in enumerate(ws):
        g = w.geom
        for tbc in ([I.dirichlet(0.3)] * len(g.tbc), [I.robin(1.0, 2.0, 0.1)] * len(g.tbc)):
            clbm.clbm_set_boundaries(changed.view(i), g.solid, tbc, g.side_tbc, g.link_node, g.link_dir, g.link_ne,
                                     g.link_tbc, g.link_q_or_half())
            # memory given back would be handed out again here
            keep += [torch.full((n,), 0x7F7F7F7F, dtype=torch.int32, device="cuda") for n in (100, 1000, 10000, 100000)]
    plain.solve(0.0, 30, 10)
    changed.solve(0.0, 30, 10)
    for i, w in enumerate(ws):
        for a, b in zip(plain.moments(i), changed.moments(i)):
            np.testing.assert_array_equal(a, b)
        clbm.clbm_step(changed.view(i), 30)  # the view's own steps take the new walls
        clbm.clbm_step(plain.view(i), 30)
        assert not np.array_equal(plain.moments(i)[3], changed.moments(i)[3])
        assert np.isfinite(changed.moments(i)[3]).all()
    plain.close()
    changed.close()
