"""Default kernel form of a single lattice, from the rule itself (host code,
compiled alone): the form's grid can be launched at every size."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GRID_Y = 65535                                     # CUDA's limit of gridDim.y
ROWS = {8: 8, 10: 4, 11: 8, 12: 4}                 # lattice rows per block of the 2-D forms


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("forms")
    src = d / "forms.cpp"
    src.write_text('#include "%s"\nextern "C" int form(const lbm_config* c) { return lbm::default_variant(c); }\n'
                   'extern "C" int batch_form(int n, const lbm_config* c) { return lbm::default_batch_variant(n, c); }\n'
                   'extern "C" int alias(int D, int single, int v) { return lbm::alias_form(D, single != 0, v); }\n'
                   'extern "C" int settled(int h, float hm, int b, float bm) { return lbm::settled_form(h, hm, b, bm); }\n'
                   % os.path.join(ROOT, "paper_2409_02930_gb300", "csrc", "lbm_forms.h"))
    so = d / "forms.so"
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


def form(rule, nx, ny, nz=1, fp64=False, bc=0):
    from paper_2409_02930_gb300 import lbm
    c = lbm.LbmConfig()
    c.nx, c.ny, c.nz, c.bc_lo, c.bc_hi = nx, ny, nz, bc, bc
    c.precision = lbm.LBM_FP64 if fp64 else lbm.LBM_FP32
    return rule.form(ctypes.byref(c))


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("bc", [0, 1, 2])
def test_default_form_can_be_launched(rule, fp64, bc):
    edges = [1, 2, 3, 65535, 65536, 4 * 65535, 4 * 65535 + 1, 8 * 65535, 8 * 65535 + 1, 600000, 4000000]
    for nx in (3, 4, 8, 20, 480):
        for ny in edges:
            if nx * ny > 2e9:
                continue
            v = form(rule, nx, ny, fp64=fp64, bc=bc)
            assert v == -1 or -(-ny // ROWS[v]) <= GRID_Y, (nx, ny, v)


def test_default_form_at_its_lines(rule):
    """Each side of every line of the rule."""
    for fp64, tile in ((False, 12), (True, 11)):
        assert form(rule, 64, 152, fp64=fp64) == 10          # 9,728 nodes
        assert form(rule, 64, 153, fp64=fp64) == tile
        assert form(rule, 4095, 2, fp64=fp64) == 10
        assert form(rule, 4096, 2, fp64=fp64) == -1
        assert form(rule, 32, 4 * 65535, fp64=fp64, bc=1) == tile
        assert form(rule, 32, 4 * 65535 + 1, fp64=fp64, bc=1) == -1
        assert form(rule, 2048, 1535, fp64=fp64) == tile
        assert form(rule, 2048, 1536, fp64=fp64) == (8 if not fp64 else tile)
        assert form(rule, 2048, 1536, fp64=fp64, bc=1) == tile
        assert form(rule, 2050, 1536, fp64=fp64) == tile
    assert form(rule, 20, 8 * 65535) == 8
    assert form(rule, 20, 8 * 65535 + 1) == -1
    assert form(rule, 12, 4, nz=4) == 5


@pytest.mark.parametrize("bc", [0, 1, 2])
def test_narrow_lattices_leave_the_tiles(rule, bc):
    """Lattices narrower than a tile run in two passes once their tiles are more
    than a few per SM, and on tiles on the other side of each line."""
    for fp64 in (False, True):
        for nx, ny in ((1, 200000), (2, 100003), (3, 66669), (4, 50003), (6, 33336), (8, 25003), (1, 9000), (1, 10000),
                       (3, 20000), (2, 5000), (4, 2500)):
            assert form(rule, nx, ny, fp64=fp64, bc=bc) == -1, (nx, ny, fp64)
    # FP32: 8 x 4 tiles up to eight per SM, 32 x 4 tiles up to four, 20 columns
    assert form(rule, 1, 4 * 1216, bc=bc) == 10
    assert form(rule, 1, 4 * 1216 + 1, bc=bc) == -1
    assert form(rule, 7, 1389, bc=bc) == 10
    assert form(rule, 16, 4 * 608, bc=bc) == 12
    assert form(rule, 16, 4 * 608 + 1, bc=bc) == -1
    assert form(rule, 19, 11000, bc=bc) == -1
    assert form(rule, 20, 11000, bc=bc) == 12
    # FP64: 8 x 4 tiles up to three per SM, 16 x 8 tiles by waves
    assert form(rule, 1, 4 * 456, fp64=True, bc=bc) == 10
    assert form(rule, 1, 4 * 456 + 1, fp64=True, bc=bc) == -1
    assert form(rule, 8, 1250, fp64=True, bc=bc) == -1
    assert form(rule, 12, 2000, fp64=True, bc=bc) == 11
    assert form(rule, 12, 16669, fp64=True, bc=bc) == -1
    assert form(rule, 14, 14288, fp64=True, bc=bc) == 11
    assert form(rule, 16, 12503, fp64=True, bc=bc) == 11
    assert form(rule, 17, 11767, fp64=True, bc=bc) == -1
    assert form(rule, 24, 1000, fp64=True, bc=bc) == 11
    assert form(rule, 31, 6454, fp64=True, bc=bc) == 11
    assert form(rule, 32, 6253, fp64=True, bc=bc) == 11


def batch_form(rule, cases, fp64=False):
    from paper_2409_02930_gb300 import lbm
    cs = (lbm.LbmConfig * len(cases))()
    for c, (nx, ny) in zip(cs, cases):
        c.nx, c.ny, c.nz = nx, ny, 1
        c.precision = lbm.LBM_FP64 if fp64 else lbm.LBM_FP32
    return rule.batch_form(len(cases), cs)


def test_batches_of_narrow_cases_leave_the_tiles(rule):
    for fp64 in (False, True):
        for nx, ny, n in ((3, 5000, 8), (4, 2000, 8), (8, 3000, 8), (12, 2000, 8), (19, 2000, 8), (3, 40000, 2)):
            assert batch_form(rule, [(nx, ny)] * n, fp64) == 0, (nx, ny, fp64)
        assert batch_form(rule, [(1000, 4)] * 64, fp64) == 10
        assert batch_form(rule, [(1000, 1)] * 64, fp64) == 0
        assert batch_form(rule, [(20, 30)], fp64) == 10
        assert batch_form(rule, [(1000, 2)] * 64, fp64) == 0
        assert batch_form(rule, [(1000, 3)] * 64, fp64) == (0 if fp64 else 10)
    assert batch_form(rule, [(20, 2000)] * 8) == 10                  # three fifths of each tile
    assert batch_form(rule, [(5, 200)] * 12) == 10                   # 600 tiles
    assert batch_form(rule, [(5, 200)] * 13) == 0
    assert batch_form(rule, [(24, 2000)] * 8, fp64=True) == 0
    assert batch_form(rule, [(29, 2000)] * 8, fp64=True) == 10       # nine tenths
    assert batch_form(rule, [(5, 200)] * 3, fp64=True) == 10         # 150 tiles
    assert batch_form(rule, [(5, 200)] * 8, fp64=True) == 0
    assert batch_form(rule, [(5, 200)] * 8 + [(2048, 256)], fp64=True) == 10


def test_alias_indices(rule):
    """Indices that a search over the forms passes over; each is one of the others."""
    for single in (0, 1):
        assert not any(rule.alias(2, single, v) for v in range(-1, 13))
        assert [v for v in range(-1, 6) if not rule.alias(3, single, v)] == ([0, 1, 2, 5] if single else [0, 1, 5])


def test_search_keeps_the_form_in_effect_on_near_ties(rule):
    rule.settled.argtypes = [ctypes.c_int, ctypes.c_float, ctypes.c_int, ctypes.c_float]
    assert rule.settled(8, 27.5, 12, 27.4) == 8
    assert rule.settled(8, 27.5, 12, 26.9) == 12
    assert rule.settled(8, 27.5, 8, 27.5) == 8
    assert rule.settled(3, 0.0, 5, 27.5) == 5                # the form in effect was not timed
