"""Edges of the kernel forms: lattices around the tile, warp and block sizes
of each form, one row and one column included, on periodic, reservoir and
bounce-back faces.

FP64 forms match the oracle to 1e-12 (field-relative per lattice), the bound
of the parity tests.  FP32 forms are held to the FP64 result of the same
steps within 16 roundings (2^-24) per step of the largest value: a node update
rounds each stored population once and its sums and products a few times more.
"""
import numpy as np
import pytest

import oracle
from paper_2409_02930_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 8
FP32_BOUND = 16 * STEPS * 2.0 ** -24


@pytest.fixture(scope="module")
def L():
    from paper_2409_02930_gb300 import lbm
    lbm.load()
    return lbm


def worst(a, b):
    return max(float(np.max(np.abs(a[k] - b[k])) / np.max(np.abs(b[k]))) for k in range(len(b)))


def slab(nx, ny, bc, energy=True):
    if bc == W.BC_INLET:
        return W.adjoint_slab(nx=nx, ny=ny, steps=STEPS)
    wl = W.slab(nx=nx, ny=ny, steps=STEPS, energy=energy)
    wl.bc_lo = wl.bc_hi = bc
    return wl


def anode(nx, ny, nz, bc_lo=W.BC_INLET, bc_hi=W.BC_BOUNCEBACK):
    return W.anode3d(nx=nx, ny=ny, nz=nz, steps=STEPS, bc_lo=bc_lo, bc_hi=bc_hi)


def check_forms(L, wl, forms):
    o = oracle.Oracle(wl)
    o.step(STEPS)
    ref = o.pops()
    for prec, bound in ((L.LBM_FP64, 1e-12), (L.LBM_FP32, FP32_BOUND)):
        for v in forms:
            g = L.Lattice(wl, precision=prec)
            g.set_variant(v)
            g.step(STEPS)
            g.sync()
            e = worst(g.populations(), ref)
            g.close()
            assert e < bound, (prec, v, e)


# around the tiles (8 x 4, 16 x 8, 32 x 4), with rows that
# wrap inside one tile (ny <= 4, 8), one row, and one node past a tile
@pytest.mark.parametrize("nx,ny,bc", [
    (3, 1, W.BC_INLET), (8, 4, W.BC_PERIODIC), (9, 5, W.BC_BOUNCEBACK), (33, 9, W.BC_INLET), (32, 8, W.BC_PERIODIC),
    (31, 7, W.BC_BOUNCEBACK), (1, 6, W.BC_PERIODIC), (40, 2, W.BC_PERIODIC), (65, 17, W.BC_INLET),
    (5, 3, W.BC_INLET)])
def test_tiles_at_their_edges(L, nx, ny, bc):
    g = L.Lattice(slab(nx, ny, bc))
    n = g.variant_count()
    g.close()
    check_forms(L, slab(nx, ny, bc), [-1] + list(range(10, n)))


@pytest.mark.parametrize("energy", [False, True])
def test_tiles_of_isothermal_and_two_species(L, energy):
    n = 13
    check_forms(L, slab(35, 10, W.BC_PERIODIC, energy), range(10, n))
    wl = W.capillary(nx=37, ny=5, steps=STEPS)
    check_forms(L, wl, range(10, n))


# 32 nodes and one warp per lattice in a block: below, at and past a block,
# faces in the middle of a warp, two layers only
@pytest.mark.parametrize("shape,bc", [
    ((3, 1, 2), (W.BC_INLET, W.BC_INLET)), ((4, 4, 2), (W.BC_PERIODIC, W.BC_PERIODIC)),
    ((11, 3, 3), (W.BC_INLET, W.BC_BOUNCEBACK)), ((2, 5, 4), (W.BC_BOUNCEBACK, W.BC_BOUNCEBACK)),
    ((33, 2, 2), (W.BC_BOUNCEBACK, W.BC_INLET))])
def test_lattice_split_3d_at_its_edges(L, shape, bc):
    check_forms(L, anode(*shape, *bc), range(0, 6))


def test_lattice_split_3d_other_mixtures(L):
    """Two and three species, with and without the energy lattice, in 3-D."""
    for M, energy in ((3, False), (3, True), (2, False)):
        wl = W.slab(nx=9, ny=5, steps=STEPS, energy=energy) if M == 3 else W.capillary(nx=9, ny=5, steps=STEPS)
        wl.nz = 3
        N = wl.nx * wl.ny * 3
        wl.porosity = np.tile(wl.porosity, 3) * np.linspace(0.8, 1.0, N)
        wl.X_init = np.tile(wl.X_init, (1, 3))
        wl.T_init, wl.P_init = np.tile(wl.T_init, 3), np.tile(wl.P_init, 3)
        check_forms(L, wl, [-1, 5])


@pytest.mark.parametrize("shape", [(3, 2, 2), (32, 16, 4), (17, 11, 11), (40, 32, 31)])
def test_surface_source_forms(L, shape):
    """A warp per node (up to 2048 nodes), a thread per node without and (past
    38,912 nodes) with a register limit, against the oracle's Newton solve:
    coverages and populations after two steps."""
    wl = W.anode3d_reactive(*shape, steps=2)
    o = oracle.Oracle(wl)
    o.step(2)
    g = L.Lattice(wl, precision=L.LBM_FP64)
    g.step(2)
    g.sync()
    assert worst(g.populations(), o.pops()) < 1e-12
    assert np.max(np.abs(g.moments(L.LBM_MOM_XS) - o.moments(oracle.MOM_XS))) < 1e-12


@pytest.mark.parametrize("ny", [1, 2, 5, 9])
def test_batch_tiles_of_ragged_cases(L, ny):
    """Cases of uneven length whose rows do not fill a tile, every batch form."""
    wls = W.capillary_batch(n_cases=5, seed=3, ny=ny, nmin=5, nmax=70, steps=STEPS)
    ref = []
    for w in wls:
        o = oracle.Oracle(w)
        o.step(STEPS)
        ref.append(o.pops())
    for v in range(12):
        b = L.Batch(wls, precision=L.LBM_FP64)
        b.set_variant(v)
        b.step(STEPS)
        b.sync()
        for p, q in zip(b.populations(), ref):
            assert worst(p, q) < 1e-12, v
        b.close()


@pytest.mark.parametrize("nx,ny,bc", [(3, 2, W.BC_INLET), (4, 1, W.BC_INLET), (2, 3, W.BC_BOUNCEBACK),
                                      (1, 3, W.BC_PERIODIC), (5, 2, W.BC_PERIODIC)])
def test_adjoint_on_degenerate_lattices(L, nx, ny, bc):
    """Every node's dJ/dphi against central differences of the oracle-exact
    FP64 forward run on lattices whose stencils fold onto themselves (both
    reservoirs share the adjacent node at nx = 3).  J is smooth and of order
    one in phi, so a step of 1e-5 leaves a truncation of 1e-9 and a rounding of
    1e-10 of the largest entry."""
    wl = slab(nx, ny, bc)
    plane = max(nx - 2, 0)
    g = L.Lattice(wl, precision=L.LBM_FP64)
    _, grad, _, _ = g.adjoint(6, 4, plane=plane)
    g.close()

    def J(phi):
        w = slab(nx, ny, bc)
        w.porosity = phi
        h = L.Lattice(w, precision=L.LBM_FP64)
        v = h.adjoint(6, 4, plane=plane)[0]
        h.close()
        return v

    eps, fd = 1e-5, np.zeros(wl.N)
    for n in range(wl.N):
        e = np.zeros(wl.N)
        e[n] = eps
        fd[n] = (J(wl.porosity + e) - J(wl.porosity - e)) / (2 * eps)
    assert np.max(np.abs(grad - fd)) <= 1e-6 * np.max(np.abs(fd)) + 1e-12


@pytest.mark.parametrize("nx,ny", [(8, 4), (37, 11)])
def test_split_2d_solves_in_double_above_the_bound(L, nx, ny):
    """The lattice-split tile (form 10) with every node's diffusion system sent
    to the FP64 solve, against the oracle within the FP32 bound."""
    wl = slab(nx, ny, W.BC_PERIODIC)
    o = oracle.Oracle(wl)
    o.step(STEPS)
    g = L.Lattice(wl, precision=L.LBM_FP32, kappa_threshold=1e-30)
    g.set_variant(10)
    g.step(STEPS)
    g.sync()
    assert worst(g.populations(), o.pops()) < FP32_BOUND
    g.close()


def test_split_2d_six_species(L):
    """Six species on a two-dimensional lattice, form 10 and the tiles."""
    check_forms(L, anode(19, 6, 1), range(10, 13))


# FP64 blocks of 8 nodes (up to 608), of 16 (up to 4864) and of 32: below, at and
# past a block and each line, species of one warp on different faces
@pytest.mark.parametrize("shape", [(3, 1, 2), (4, 2, 3), (38, 4, 4), (29, 7, 3), (203, 3, 8), (32, 19, 8),
                                   (139, 7, 5)])
def test_small_blocks_3d(L, shape):
    wl = anode(*shape)
    o = oracle.Oracle(wl)
    o.step(2)
    g = L.Lattice(wl, precision=L.LBM_FP64)
    g.step(2)
    g.sync()
    assert worst(g.populations(), o.pops()) < 1e-12
    g.close()


@pytest.mark.parametrize("steps", [1, 2, 7])
def test_surface_source_of_low_rank_mechanisms(L, steps):
    """The first steps of the mechanism only: one independent change, a step and
    its reverse, and species that take no part; a warp and a thread per node."""
    mc = W.surface_mechanism()
    for k in ("nu_gas", "nu_surf", "A", "Ea"):
        setattr(mc, k, np.ascontiguousarray(getattr(mc, k)[:steps]))
    mc.R = steps
    for shape in ((4, 2, 2), (17, 11, 11)):
        wl = W.anode3d(*shape, mechanism=mc, steps=2)
        o = oracle.Oracle(wl)
        o.step(2)
        g = L.Lattice(wl, precision=L.LBM_FP64)
        g.step(2)
        g.sync()
        assert worst(g.populations(), o.pops()) < 1e-12
        assert np.max(np.abs(g.moments(L.LBM_MOM_XS) - o.moments(oracle.MOM_XS))) < 1e-12
        g.close()


@pytest.mark.parametrize("shape", [(7, 4, 3), (33, 9, 5), (21, 18, 16)])
def test_indices_that_are_one_form(L, shape):
    """D3Q27 indices that name one form return the same bits, and the autotuner
    settles on one of the forms that differ."""
    wl = anode(*shape)
    for prec in (L.LBM_FP64, L.LBM_FP32):
        pops = {}
        for v in (-1, 0, 1, 2, 3, 4, 5):
            g = L.Lattice(wl, precision=prec)
            g.set_variant(v)
            g.step(2)
            g.sync()
            pops[v] = g.populations()
            g.close()
        same = [(-1, 5), (3, 5), (4, 5)] + ([(1, 2)] if prec == L.LBM_FP64 else [])
        assert all(np.array_equal(pops[a], pops[b]) for a, b in same)
        g = L.Lattice(wl, precision=prec)
        assert g.autotune(2) in ((0, 1, 2, 5) if prec == L.LBM_FP32 else (0, 1, 5))
        g.close()


# a warp per node up to 7,296 (FP32) and 4,864 (FP64) nodes, one past the line,
# and inside the thread form without a register limit
@pytest.mark.parametrize("shape,precision", [((19, 16, 16), "fp64"), ((17, 41, 7), "fp64"), ((32, 16, 12), "fp64"),
                                             ((19, 24, 16), "fp32"), ((8, 48, 20), "fp32"), ((24, 20, 18), "fp32")])
def test_surface_source_at_its_lines(L, shape, precision):
    """FP64 within the parity bound; in FP32 the populations within 16 roundings a
    step and the coverages, which are FP64, within 1e-8, the bound of the tests at
    full size."""
    wl = W.anode3d_reactive(*shape, steps=2)
    o = oracle.Oracle(wl)
    o.step(2)
    fp64 = precision == "fp64"
    g = L.Lattice(wl, precision=L.LBM_FP64 if fp64 else L.LBM_FP32)
    g.step(2)
    g.sync()
    assert worst(g.populations(), o.pops()) < (1e-12 if fp64 else 16 * 2 * 2.0 ** -24)
    assert np.max(np.abs(g.moments(L.LBM_MOM_XS) - o.moments(oracle.MOM_XS))) < (1e-12 if fp64 else 1e-8)
    g.close()


@pytest.mark.parametrize("steps", [1, 7])
def test_thread_form_of_low_rank_mechanisms(L, steps):
    """As test_surface_source_of_low_rank_mechanisms, on a lattice above the warp
    form's line."""
    mc = W.surface_mechanism()
    for k in ("nu_gas", "nu_surf", "A", "Ea"):
        setattr(mc, k, np.ascontiguousarray(getattr(mc, k)[:steps]))
    mc.R = steps
    wl = W.anode3d(17, 41, 7, mechanism=mc, steps=2)
    o = oracle.Oracle(wl)
    o.step(2)
    g = L.Lattice(wl, precision=L.LBM_FP64)
    g.step(2)
    g.sync()
    assert worst(g.populations(), o.pops()) < 1e-12
    assert np.max(np.abs(g.moments(L.LBM_MOM_XS) - o.moments(oracle.MOM_XS))) < 1e-12
    g.close()
