"""Lattices with more rows than a row-tiled form's grid can count: the default
form steps them, the forms that cannot say so and leave the context usable, and
the others agree with the two-pass form."""
import numpy as np
import pytest

from paper_2409_02930_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BOUND = 16 * 2 * 2.0 ** -24            # initial equilibria and one step, 16 roundings each


def test_more_rows_than_a_grid_counts():
    from paper_2409_02930_gb300 import lbm as L
    wl = W.slab(nx=4, ny=8 * 65535 + 1, steps=1)
    g = L.Lattice(wl, precision=L.LBM_FP32)
    assert g.variant() == -1
    p0 = g.populations()
    g.step(1)
    g.sync()
    ref = g.populations()
    ran = []
    for v in range(g.variant_count()):
        g.set_populations(p0)
        g.set_variant(v)
        try:
            g.step(1)
        except L.LbmError as e:
            assert "cannot run this lattice" in str(e)
            continue
        g.sync()
        ran.append(v)
        for a, b in zip(g.populations(), ref):
            assert np.max(np.abs(a - b)) < BOUND * np.max(np.abs(b)), v
    # the march of 16 rows a block and the forms with a flat grid
    assert ran == [4, 6, 7], ran
    g.set_populations(p0)
    g.set_variant(-1)
    g.step(1)
    g.sync()
    assert np.array_equal(g.populations(), ref)
    assert g.autotune(1) in [-1] + ran
    g.close()
