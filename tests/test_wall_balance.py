"""Walls of given flux (b2 = 0) keep the heat of a uniform temperature: their
weights, as rounded, sum to the share of it that the collision, with its
constants as rounded, keeps in an axis pair."""
import ctypes as C
import itertools
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("balance") / "libbalance.so")
    r = subprocess.run([nvcc, "-shared", "-Xcompiler", "-fPIC", "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                        "-gencode", "arch=compute_103a,code=sm_103a", "-o", out, os.path.join(HERE, "host_balance.cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(out)
    d = C.c_double
    L.host_round_heat.argtypes = [d, d, d, d, d, C.c_int, C.c_int, d, d, C.POINTER(d)]
    return L


FRACTIONS = [1e-3, 0.2, 0.5 - 1e-9, 0.5, 0.5 + 1e-9, 0.77, 1.0]


@pytest.mark.parametrize("cT2", [0.4, 1.0 / 3.0, 0.25, 0.1, 0.49])
@pytest.mark.parametrize("l2", [0.05, 0.7, 1.1, 1.95])
def test_flux_walls_balance(harness, cT2, l2):
    k = (C.c_double * 10)()
    for b1, b3, q, have2 in itertools.product((1.0, 0.3, 7.0), (0.0, 0.03), FRACTIONS, (0, 1)):
        harness.host_round_heat(b1, 0.0, b3, 0.9, q, have2, 1, l2, cT2, k)
        for off, R in ((0, np.float64), (5, np.float32)):
            eps = float(np.finfo(R).eps)
            # the collision's fixed point G20 = (1 - l2) / 2 x 2 G20 + l2 cT2 / 2, constants rounded to R
            a, s = Fraction(float(R(0.5 * (1.0 - l2)))), Fraction(float(R(0.5 * l2 * cT2)))
            share = 2 * s / (1 - 2 * a)
            assert abs(float(share) - k[off + 4]) <= 4e-16 / l2
            w = [k[off + m] for m in (0, 1, 3)]
            assert w[2] == 0
            if have2:  # |w1| <= cT2 / 4: half an ulp of it is at most eps cT2 / 8
                assert abs(float(Fraction(w[0]) + Fraction(w[1]) - share)) <= eps * cT2 / 8 + 4e-16 / l2
            else:  # one weight: the nearest number
                assert w[1] == 0 and abs(float(Fraction(w[0]) - share)) <= eps * cT2 / 2 + 4e-16 / l2


def test_other_walls_are_rounded_one_by_one(harness):
    k = (C.c_double * 10)()
    for (b1, b2), q, have2, have3 in itertools.product([(0.0, 1.0), (1.0, 0.4), (2.5, 1e-3)], FRACTIONS, (0, 1), (0, 1)):
        harness.host_round_heat(b1, b2, 0.2, 0.9, q, have2, have3, 1.1, 0.4, k)
        for m in range(4):
            assert np.float32(k[m]) == k[5 + m]


@pytest.mark.parametrize("l2", [1e-3, 1e-4, 1e-6, 1e-8, 1e-12, 1e-17])
def test_small_rates(harness, l2):
    """The rounded constants of a rate near zero say nothing about the share (1 - l2
    may round to 1): the weights stay at cT2."""
    k = (C.c_double * 10)()
    for q, have2 in itertools.product(FRACTIONS, (0, 1)):
        harness.host_round_heat(1.0, 0.0, 0.1, 0.9, q, have2, 0, l2, 0.4, k)
        for off, R in ((0, np.float64), (5, np.float32)):
            assert abs(k[off] + k[off + 1] - 0.4) <= 1026 * float(np.finfo(R).eps) * 0.4, (q, have2, R)
