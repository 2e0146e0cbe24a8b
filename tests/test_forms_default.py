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
                   % os.path.join(ROOT, "paper_2409_02930_gb300", "csrc", "lbm_forms.h"))
    so = d / "forms.so"
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so)).form


def form(rule, nx, ny, nz=1, fp64=False, bc=0):
    from paper_2409_02930_gb300 import lbm
    c = lbm.LbmConfig()
    c.nx, c.ny, c.nz, c.bc_lo, c.bc_hi = nx, ny, nz, bc, bc
    c.precision = lbm.LBM_FP64 if fp64 else lbm.LBM_FP32
    return rule(ctypes.byref(c))


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
        assert form(rule, 4, 4 * 65535, fp64=fp64) == tile
        assert form(rule, 4, 4 * 65535 + 1, fp64=fp64) == -1
        assert form(rule, 2048, 1535, fp64=fp64) == tile
        assert form(rule, 2048, 1536, fp64=fp64) == (8 if not fp64 else tile)
        assert form(rule, 2048, 1536, fp64=fp64, bc=1) == tile
        assert form(rule, 2050, 1536, fp64=fp64) == tile
    assert form(rule, 8, 8 * 65535) == 8
    assert form(rule, 8, 8 * 65535 + 1) == -1
    assert form(rule, 12, 4, nz=4) == 5
