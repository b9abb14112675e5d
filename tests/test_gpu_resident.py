"""Steps taken in shared memory (many steps a launch) and tiles with inline
walls, against the plane kernels' single steps with listed boundary nodes.

Every kernel that updates a node rounds at the same points, so the comparisons
are bit for bit."""
import dataclasses

import numpy as np
import pytest

from paper_1801_04577_gb300 import clbm
from paper_1801_04577_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def lattices():
    return {
        "cavity24": I.natural_convection_cavity(24, 1e4),
        "cavity33": I.natural_convection_cavity(33, 1e4),       # bands of 2 and 3 rows
        "cavity128": I.natural_convection_cavity(128, 1e4),
        "rows31": I.rayleigh_benard(40, 31, Ra=1e4, noise=1e-2),  # fewer bands than 16
        "rows2": I.rayleigh_benard(70, 2, Ra=1e4, noise=1e-2),
        "periodic": I.periodic_box(29, 34),                      # the seam joins the first and last band
        "one_row": I.periodic_box(33, 1),                        # its own neighbour on both sides
        "one_column": I.couette_channel(19, nx=1),
        "channel": I.obstacle_channel(61, 37),
        "annulus": I.annulus(64, 2.6, Ra=1e4),
        "interpolated": I.annulus(64, 2.6, Ra=1e4, interpolated=True),
        "couette_vh": I.couette_channel(16, nx=9, viscous_heating=1),
    }


@pytest.mark.parametrize("precision,rounding", [("f32", 0), ("f16", 1), ("bf16", 0), ("f64", 0)])
@pytest.mark.parametrize("name", sorted(lattices()))
def test_many_steps_equal_single_steps(name, precision, rounding):
    w = lattices()[name]
    a = clbm.from_workload(w, precision, rounding=rounding)
    b = clbm.from_workload(w, precision, rounding=rounding)
    for n in (7, 2, 12):  # odd, shortest, even: the buffers alternate
        a.step(n)
        for _ in range(n):
            b.step(1)
    assert a.time == b.time == 21
    for x, y in zip(a.moments(), b.moments()):
        np.testing.assert_array_equal(x, y)
    assert a.residual() == b.residual()  # both states are there
    a.step(1)
    b.step(1)
    for x, y in zip(a.moments(), b.moments()):
        np.testing.assert_array_equal(x, y)


SIZES = [(1, 3), (2, 2), (3, 1), (31, 4), (33, 3), (63, 2), (64, 5), (127, 3), (128, 3), (129, 4), (130, 2),
         (511, 2), (513, 3), (645, 2)]


@pytest.mark.parametrize("precision,rounding", [("f32", 0), ("f64", 0), ("f16", 1), ("bf16", 0)])
@pytest.mark.parametrize("walls", ["box", "periodic_x", "periodic_y", "periodic"])
def test_inline_walls_equal_listed_nodes(walls, precision, rounding):
    """A box lattice (walls and seams inside the tiles) against the same one
    with an empty mask (edge nodes from the list), one step a launch, at rows
    around the ends of tiles, vectors and blocks, and fewest rows."""
    px, py = walls in ("periodic_x", "periodic"), walls in ("periodic_y", "periodic")
    tbc = [I.dirichlet(1.0), I.robin(1.0, 0.5, 0.1), I.neumann(0.02), I.robin(2.0, 0.3, 0.2)]
    for nx, ny in SIZES:
        p = I.Params(nx=nx, ny=ny, periodic_x=int(px), periodic_y=int(py), s_nu=1.2, lambda1=1.3, T0=0.5,
                     gbeta=2e-4, Q=3e-5, Fvx=1e-5)
        g = I.Geometry(tbc=tbc, side_tbc=(-1 if px else 0, -1 if px else 1, -1 if py else 2, -1 if py else 3))
        init = I.random_fields(nx, ny, 11, amp=0.01)
        masked = dataclasses.replace(g, solid=np.zeros((ny, nx), np.uint8))
        out = []
        for geom in (g, masked):
            s = clbm.Solver(p, geom, precision, None, init, rounding)
            for _ in range(5):
                s.step(1)
            out.append(s.moments())
            s.close()
        for x, y in zip(*out):
            np.testing.assert_array_equal(x, y, err_msg=f"{nx}x{ny}")


@pytest.mark.parametrize("precision,rounding", [("f32", 0), ("f16", 1)])
def test_batched_lattices_equal_single_steps(precision, rounding):
    """Lattices of a batch by every route: resident in half and in all of a
    multiprocessor's memory, tiles with inline walls, tiles with a mask."""
    ws = I.obstacle_cavities(2, 128) + I.obstacle_cavities(1, 48) + [I.rayleigh_benard(600, 90, Ra=1e5, noise=1e-2),
                                                                    I.obstacle_channel(700, 120)]
    b = clbm.Batch(ws, precision, rounding=rounding)
    conv, _, steps = b.solve(0.0, 20, check_every=10)
    assert steps == 20 and (conv == -1).all()
    for i, w in enumerate(ws):
        s = clbm.from_workload(w, precision, rounding=rounding)
        for _ in range(20):
            s.step(1)
        for x, y in zip(b.moments(i), s.moments()):
            np.testing.assert_array_equal(x, y, err_msg=w.name)
        s.close()
    b.close()
