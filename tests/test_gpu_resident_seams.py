"""Off-midpoint Dirichlet walls beside the seam of a periodic y axis: steps of
any route against single steps, bit for bit, and against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_1801_04577_gb300 import clbm
from paper_1801_04577_gb300 import inputs as I

from _parity import TOL, compare

pytestmark = pytest.mark.gpu

NX, NY, RADIUS = 24, 26, 4.3


def cylinder(cy):
    """A doubly periodic box with a heated cylinder centred at (11.4, cy): every
    link into it at the fraction where it crosses the circle (both below and above 1/2)."""
    cx = 11.4
    wrap = lambda d, n: (d + n / 2) % n - n / 2  # noqa: E731
    X = wrap(np.arange(NX)[None, :] - cx, NX) + np.zeros((NY, 1))
    Y = wrap(np.arange(NY)[:, None] - cy, NY) + np.zeros((1, NX))
    solid = (X * X + Y * Y < RADIUS * RADIUS).astype(np.uint8)
    nodes, dirs, nes, tbcs, qs = [], [], [], [], []
    for y, x in zip(*np.nonzero(solid == 0)):
        for d in range(1, 9):
            if not solid[(y + I.EY[d]) % NY, (x + I.EX[d]) % NX]:
                continue
            px, py, e2 = X[y, x], Y[y, x], I.EX[d] ** 2 + I.EY[d] ** 2
            pe = (px * I.EX[d] + py * I.EY[d]) / e2
            s = -pe - np.sqrt(pe * pe - (px * px + py * py - RADIUS ** 2) / e2)
            s = min(max(s, 1e-3), 1.0)
            ne = -((px + s * I.EX[d]) * I.EX[d] + (py + s * I.EY[d]) * I.EY[d]) / RADIUS
            nodes.append(y * NX + x), dirs.append(d), qs.append(s)
            nes.append(max(ne, 1e-3) if d <= 4 else 0.0), tbcs.append(0 if d <= 4 else -1)
    s_nu, lambda1 = I.rates_from_diffusivities(0.05, 0.06)
    p = I.Params(nx=NX, ny=NY, periodic_x=1, periodic_y=1, s_nu=s_nu, lambda1=lambda1, T0=0.5, gbeta=2e-4, Q=1e-5)
    order = np.lexsort((dirs, nodes))
    g = I.Geometry(tbc=[I.dirichlet(1.0)], side_tbc=(-1, -1, -1, -1), solid=solid,
                   link_node=np.asarray(nodes, np.int32)[order], link_dir=np.asarray(dirs, np.int32)[order],
                   link_ne=np.asarray(nes)[order], link_tbc=np.asarray(tbcs, np.int32)[order],
                   link_q=np.asarray(qs)[order])
    vertical = np.isin(g.link_dir, (2, 4)) & (g.link_q < 0.5)
    assert vertical.any()
    return I.Workload(f"cylinder{cy}", p, g, I.random_fields(NX, NY, 5, amp=0.01))


# the cylinder's edge no, one, two and three rows from the seam, on either side of it, and across it
CENTRES = (13.0, 4.6, 5.6, 6.6, 20.4, 19.4, 18.4, 0.3, 25.2)


@pytest.mark.parametrize("precision,rounding", [("f32", 0), ("f16", 1), ("bf16", 0), ("f64", 0)])
@pytest.mark.parametrize("cy", CENTRES)
def test_walls_beside_the_seam(cy, precision, rounding):
    w = cylinder(cy)
    a, b = (clbm.from_workload(w, precision, rounding=rounding) for _ in range(2))
    batch = clbm.Batch([w, cylinder(13.0)], precision, rounding=rounding)
    for n in (7, 13):
        a.step(n)
        for _ in range(n):
            b.step(1)
    batch.solve(0.0, 20, check_every=10)
    for x, y, z in zip(a.moments(), b.moments(), batch.moments(0)):
        np.testing.assert_array_equal(x, y)
        np.testing.assert_array_equal(z, y)
    assert a.residual() == b.residual()
    if precision in ("f64", "f32"):
        o = oracle.from_workload(w)
        o.step(20)
        errs = compare(w, a.moments(), o.moments(), floor=True)  # 20 steps from nearly rest
        assert max(errs.values()) <= TOL[precision], errs
    for s in (a, b, batch):
        s.close()
