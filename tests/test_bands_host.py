"""Where the rule of an off-midpoint Dirichlet link (q < 1/2) finds its third
node, against the rows that a block of the resident steps holds."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
EY = (0, 0, 1, 0, -1)


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = str(tmp_path_factory.mktemp("bands") / "libbands.so")
    r = subprocess.run([nvcc, "-shared", "-Xcompiler", "-fPIC", "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                        "-gencode", "arch=compute_103a,code=sm_103a", "-o", out, os.path.join(HERE, "host_bands.cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(out)
    L.host_reads_third.argtypes = [C.c_int, C.c_double, C.c_double]
    L.host_heat_entry.restype = L.host_bounce_entry.restype = C.c_longlong
    return L


def test_which_links_read_a_third_node(harness):
    for d in range(1, 9):
        assert harness.host_reads_third(d, 0.3, 0.0) == (d <= 4)
        assert not harness.host_reads_third(d, 0.5, 0.0)
        assert not harness.host_reads_third(d, 0.3, 1.0)


@pytest.mark.parametrize("py", [0, 1])
@pytest.mark.parametrize("ny", [1, 2, 3, 4, 7, 30])
def test_one_band_reads_only_its_own_rows(harness, ny, py):
    """One band stores the lattice's rows as local rows 1 .. ny between two
    ghost rows, and a neighbour is the local row without wrapping: an accepted
    link's third node must be one of rows 1 .. ny, or (y walls) not exist."""
    for y in range(ny):
        for d in (1, 2, 3, 4):
            local = y + 1 - 2 * EY[d]  # the link points at the wall: the third node lies the other way
            assert harness.host_third_row(y, d) == local - 1
            exists = py or 0 <= local - 1 < ny
            ok = harness.host_band_holds_third(y, d, ny, 1, py)
            assert ok == (not exists or 1 <= local <= ny)


def test_several_bands_are_refused(harness):
    assert not any(harness.host_band_holds_third(y, d, 32, cl, py)
                   for y in range(32) for d in (1, 2, 3, 4) for cl in (2, 4, 8, 16) for py in (0, 1))


@pytest.mark.parametrize("py", [0, 1])
@pytest.mark.parametrize("NY,y0,rows", [(9, 0, 9), (9, 0, 1), (9, 0, 2), (9, 3, 1), (9, 3, 2), (9, 3, 3), (9, 7, 2), (2, 1, 1)])
def test_slabs_hold_the_third_node_or_refuse(harness, NY, y0, rows, py):
    """A slab stores lattice rows y0 - 1 .. y0 + rows (around the seam of a
    periodic axis).  The third node of a link lies two rows away from the wall."""
    stored = range(y0 - 1, y0 + rows + 1)
    for gy in range(y0, y0 + rows):
        for d in (1, 2, 3, 4):
            g3 = gy - 2 * EY[d]
            none = not py and not 0 <= g3 < NY
            ok = harness.host_slab_holds_third(gy - y0 + 1, gy, d, rows + 2, NY, py)
            assert ok == (none or g3 in stored), (gy, d)


def test_link_table_entries_of_large_lattices(harness):
    """Every entry its own place, also beyond 2^31 coefficients."""
    for slot in (0, 1, 89478486, 134217728, 178956970, 2 ** 28 - 2):
        heat = [harness.host_heat_entry(s, d) for s in (slot, slot + 1) for d in (1, 2, 3, 4)]
        assert heat == list(range(16 * slot, 16 * (slot + 2), 4))
        bounce = [harness.host_bounce_entry(s, d) for s in (slot, slot + 1) for d in range(1, 9)]
        assert bounce == list(range(24 * slot, 24 * (slot + 2), 3))
