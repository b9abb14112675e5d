"""The coefficients that the step kernels take for a wall link, against the
wall profile solved in exact rationals, over every kind of wall."""
import ctypes as C
import itertools
import os
import shutil
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("walls") / "libwalls.so")
    r = subprocess.run([nvcc, "-shared", "-Xcompiler", "-fPIC", "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                        "-gencode", "arch=compute_103a,code=sm_103a", "-o", out, os.path.join(HERE, "host_walls.cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(out)
    d = C.c_double
    L.host_link_heat.argtypes = [d, d, d, d, d, C.c_int, C.c_int, d, d, d, C.POINTER(d)]
    L.host_link_bounce.argtypes = [d, C.c_int, C.POINTER(d)]
    return L


WALLS = [(0.0, 1.0, 0.7), (1.0, 0.0, 0.0), (1.0, 0.0, 0.03), (1.0, 0.4, 0.2), (2.5, 1e-3, -0.1)]
FRACTIONS = [1e-3, 0.2, 0.5 - 1e-9, 0.5, 0.5 + 1e-9, 0.8, 1.0]


def midpoint(b1, b2, b3, ne, q, T1, T2, T3, have2, have3):
    """T at s = q - 1/2 of the wall profile: Lagrange's polynomial through the
    nodes, with the wall value that solves b1 dT/dn + b2 T = b3, dT/dn = -T'(0) / ne."""
    def lagrange(xs, x):
        return [np.prod([(x - b) / (a - b) for b in xs if b != a]) for a in xs]

    def slope(xs):  # T'(0) of the same polynomials: weights
        return [sum(np.prod([-b / (a - b) for b in xs if b not in (a, c)] or [F(1)]) / (a - c) for c in xs if c != a)
                for a in xs]

    b1, b2, b3, ne, q, T1, T2, T3 = (F(v) for v in (b1, b2, b3, ne, q, T1, T2, T3))
    xs, T = ([F(0), q, 1 + q], [T1, T2]) if have2 else ([F(0), q], [T1])
    d = slope(xs)
    # b1 (-(d0 Tw + d.T) / ne) + b2 Tw = b3
    Tw = (b3 + b1 / ne * sum(a * b for a, b in zip(d[1:], T))) / (b2 - b1 * d[0] / ne)
    if b1 == 0 and q < F(1, 2):
        xs, T = ([F(0), 1 + q, 2 + q], [T2, T3]) if have2 and have3 else ([F(0), 1 + q], [T2]) if have2 else ([F(0)], [])
        if not T:
            return Tw
    return sum(a * b for a, b in zip(lagrange(xs, q - F(1, 2)), [Tw] + T))


def test_link_heat_matches_the_wall_rules(harness):
    """cT2 (T_m - T0) from the profile, and from the coefficients applied
    to s = T - T0 + Q/2.  Bound: a few dozen roundings of values up to the
    largest coefficient (1 / q)."""
    rng = np.random.RandomState(3)
    T0, hQ, cT2 = 0.5, 2e-5, 0.4
    k = (C.c_double * 4)()
    for (b1, b2, b3), q, have2, have3 in itertools.product(WALLS, FRACTIONS, (0, 1), (0, 1)):
        ne = 0.2 + 0.8 * rng.rand()
        T1, T2, T3 = 0.5 + 0.5 * (2 * rng.rand(3) - 1)
        harness.host_link_heat(b1, b2, b3, ne, q, have2, have3, T0, hQ, cT2, k)
        Tm = float(midpoint(b1, b2, b3, ne, q, T1, T2, T3, have2, have3))
        s1, s2, s3 = (T - T0 + hQ for T in (T1, T2, T3))
        got = k[0] * s1 + k[1] * s2 + k[3] * s3 + k[2]
        scale = cT2 * (1 + max(abs(v) for v in k) / cT2)
        assert abs(got - cT2 * (Tm - T0)) <= 1e-14 * scale, (b1, b2, b3, ne, q, have2, have3)
        if not have2:
            assert k[1] == 0.0 and k[3] == 0.0  # nothing is read there
        if not have3:
            assert k[3] == 0.0


def test_link_bounce(harness):
    k = (C.c_double * 3)()
    for q, have2 in itertools.product(FRACTIONS, (0, 1)):
        harness.host_link_bounce(q, have2, k)
        if q == 0.5 or (q < 0.5 and not have2):
            assert tuple(k) == (1.0, 0.0, 0.0)
        elif q < 0.5:
            np.testing.assert_allclose(k[:], [2 * q, 1 - 2 * q, 0], rtol=1e-15)
        else:
            np.testing.assert_allclose(k[:], [1 / (2 * q), 0, (2 * q - 1) / (2 * q)], rtol=1e-15)
