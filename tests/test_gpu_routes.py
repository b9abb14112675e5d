"""Which steps a lattice takes in shared memory, as the library reports it, at
the ends of the rule's ranges; every route gives single steps bit for bit."""
import numpy as np
import pytest

from paper_1801_04577_gb300 import clbm
from paper_1801_04577_gb300 import inputs as I

from test_gpu_resident_seams import cylinder

pytestmark = pytest.mark.gpu


def plane_launches(n):
    """One a step, the counter, and the graphs of 32, 16, ..., 2 steps."""
    return n if n < 2 else n + 1 + n // 32 + bin((n % 32) >> 1).count("1")


CASES = [
    # lattice, precision, rounding, steps, resident
    (lambda: I.natural_convection_cavity(64, 1e4), "f32", 0, 2, False),   # 256 nodes a band: from 3 steps on
    (lambda: I.natural_convection_cavity(64, 1e4), "f32", 0, 3, True),
    (lambda: I.natural_convection_cavity(32, 1e4), "f64", 0, 5, True),    # 64 nodes a band
    (lambda: I.natural_convection_cavity(33, 1e4), "f64", 0, 5, False),
    (lambda: I.annulus(20, 2.6, Ra=1e4), "f64", 0, 7, True),              # a mask, eight bands of up to 60 nodes
    (lambda: I.annulus(24, 2.6, Ra=1e4), "f64", 0, 7, False),             # ... of 72
    (lambda: I.obstacle_channel(16, 61), "f64", 0, 7, True),
    (lambda: I.annulus(24, 2.6, Ra=1e4, interpolated=True), "f32", 0, 9, True),  # off the midpoint: one band
    (lambda: I.annulus(32, 2.6, Ra=1e4, interpolated=True), "f32", 0, 9, True),
    (lambda: I.annulus(32, 2.6, Ra=1e4, interpolated=True), "f32", 0, 7, False),
    (lambda: I.annulus(48, 2.6, Ra=1e4, interpolated=True), "f32", 0, 40, False),  # beyond a block's memory
    (lambda: I.annulus(48, 2.6, Ra=1e4, interpolated=True), "f16", 0, 19, True),   # 256 boundary nodes
    (lambda: I.annulus(52, 2.6, Ra=1e4, interpolated=True), "bf16", 0, 40, False),
    (lambda: I.annulus(44, 2.6, Ra=1e4, interpolated=True), "f16", 1, 25, True),
    (lambda: I.annulus(48, 2.6, Ra=1e4, interpolated=True), "f16", 1, 40, False),  # stochastic: 1950 nodes
    (lambda: I.obstacle_channel(200, 150), "f16", 0, 17, True),
    (lambda: I.obstacle_channel(200, 150), "f16", 1, 40, False),
    (lambda: cylinder(13.0), "f32", 0, 11, True),
    (lambda: cylinder(4.6), "f32", 0, 11, False),   # a third node across the seam
    (lambda: cylinder(19.4), "bf16", 0, 11, False),
]


@pytest.mark.parametrize("k", range(len(CASES)))
def test_route_and_result(k):
    make, precision, rounding, n, resident = CASES[k]
    w = make()
    a, b = (clbm.from_workload(w, precision, rounding=rounding) for _ in range(2))
    assert a.step_launches(n) == (1 if resident else plane_launches(n))
    assert a.step_launches(1) == 1 and a.step_launches(0) == 0
    if resident:
        assert a.step_launches(10000) == 3
    for m in (n, n + 1):
        a.step(m)
        for _ in range(m):
            b.step(1)
    for x, y in zip(a.moments(), b.moments()):
        np.testing.assert_array_equal(x, y)
    assert a.residual() == b.residual()
    a.close()
    b.close()


def test_batch_launches():
    C = I.natural_convection_cavity
    small, masked, wide, obstacle = C(32, 1e4), I.obstacle_channel(500, 120), C(400, 1e4), I.obstacle_cavities(1, 32)[0]
    for ws, precision, K, want in (([small] * 4, "f32", 12, (1, 0, 5)),        # one cluster size
                                   ([small] * 4, "f32", 10, (0, 1, 5)),        # from intervals of 12 on,
                                   ([obstacle] * 4, "f32", 6, (1, 0, 5)),      # with a mask of 6
                                   ([obstacle] * 4, "f32", 3, (0, 2, 5)),      # tiles and their boundary nodes
                                   ([small] * 4, "f64", 100, (0, 1, 5)),
                                   ([wide, masked], "f32", 100, (0, 3, 5)),    # without and with a mask
                                   ([small, wide], "f32", 100, (1, 1, 5)),
                                   ([small, wide, obstacle], "f32", 8, (1, 1, 5)),
                                   ([small, wide, obstacle], "f32", 4, (0, 3, 5)),
                                   ([small, wide, obstacle], "f32", 12, (2, 1, 5))):
        b = clbm.Batch(ws, precision, autotune=False)
        assert b.launches(K) == want, (precision, K)
        b.close()


@pytest.mark.parametrize("precision,rounding", [("f32", 0), ("f16", 1)])
def test_check_intervals_do_not_change_results(precision, rounding):
    """Every kind of lattice by the routes that intervals of 2 .. 24 steps choose."""
    ws = [I.natural_convection_cavity(32, 1e4), I.obstacle_cavities(1, 32)[0], I.natural_convection_cavity(300, 1e4),
          I.obstacle_cavities(1, 128)[0], I.obstacle_channel(500, 120)]
    b = clbm.Batch(ws, precision, rounding=rounding)
    start = [[np.copy(a) for a in b.moments(i)] for i in range(len(ws))]
    want = None
    for K in (24, 12, 8, 6, 4, 2, 24):
        for i, m in enumerate(start):
            clbm.clbm_init_fields(b.view(i), *m)
        conv, _, steps = b.solve(0.0, 24, K)
        assert steps == 24 and (conv == -1).all()
        got = [b.moments(i) for i in range(len(ws))]
        if want is None:
            want = got
        for x, y in zip(got, want):
            for p, q in zip(x, y):
                np.testing.assert_array_equal(p, q, err_msg=str(K))
    b.close()
