"""Slabs and off-midpoint Dirichlet links: a slab that does not store a link's
third node is refused; accepted partitions equal the whole lattice bit for bit."""
import numpy as np
import pytest

from paper_1801_04577_gb300 import clbm
from paper_1801_04577_gb300 import inputs as I
from paper_1801_04577_gb300 import slabs

pytestmark = pytest.mark.gpu


def missing(w, y0, rows):
    """Links of the slab's rows whose third node (two rows from the node, away
    from the wall) is a row of the lattice that the slab does not store."""
    g, ny = w.geom, w.params.ny
    out = 0
    for node, d, t, q in zip(g.link_node, g.link_dir, g.link_tbc, g.link_q):
        y = node // w.params.nx
        if not (y0 <= y < y0 + rows and d in (2, 4) and q < 0.5 and g.tbc[t][0] == 0.0):
            continue
        y3 = y - 2 * I.EY[d]
        if not w.params.periodic_y and not 0 <= y3 < ny:
            continue
        out += not y0 - 1 <= y3 <= y0 + rows
    return out


def lattices():
    """Walls above and below their nodes: the heated cylinder of an annulus, a
    channel whose bottom (q < 1/2) or top wall lies off the midpoint."""
    w = {"annulus": I.annulus(24, 2.6, Ra=1e4, interpolated=True), "bottom": I.offset_channel(10, 0.3, 0.8),
         "top": I.offset_channel(10, 0.8, 0.3)}
    for v in w.values():
        v.init = I.random_fields(v.params.nx, v.params.ny, 3, amp=0.01)
    return w


@pytest.mark.parametrize("precision,rounding", [("f32", 0), ("f16", 1)])
@pytest.mark.parametrize("name", ["annulus", "bottom", "top"])
def test_thin_slabs(name, precision, rounding):
    w = lattices()[name]
    ref = clbm.from_workload(w, precision, rounding=rounding)
    for _ in range(20):
        ref.step(1)
    want, accepted = ref.moments(), 0
    for parts in range(1, w.params.ny + 1):
        if any(missing(w, y0, rows) for y0, rows in slabs.partition(w.params.ny, parts)):
            with pytest.raises(clbm.ClbmError) as e:
                slabs.SlabGroup(w, parts, precision, rounding)
            assert e.value.status == clbm.CLBM_EINVAL
            continue
        accepted += 1
        g = slabs.SlabGroup(w, parts, precision, rounding)
        g.step(20)
        for a, b in zip(g.moments(), want):
            np.testing.assert_array_equal(a, b, err_msg=f"{parts} slabs")
        g.close()
    assert 0 < accepted < w.params.ny
    ref.close()
