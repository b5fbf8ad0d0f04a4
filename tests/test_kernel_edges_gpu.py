"""Edges of the kernels' thread layouts against the FP64 oracle: the smallest
and largest band counts, direction counts and grids each layout accepts.  The
bars are those of the FP64 parity tests: T to rel 1e-12, I to rel 1e-11."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_19400_gb300 import bte, workloads as W

pytestmark = pytest.mark.gpu


def workload(shape, dirs, bands, kinds, temps, dt=1e-12, nsteps=2, ninner=4):
    nx, ny, nz = shape
    g = W.Geometry(2 if nz == 1 else 3, nx, ny, nz, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, kinds, temps)
    return W.Workload("edges", [g], dirs, W.make_bands(*bands), dt, nsteps, ninner)


def check(wl, s, scheme=O.IMPLICIT, T0=None, dt=None):
    """The solver's state after wl.nsteps against the oracle's."""
    g = wl.geoms[0]
    p = O.Problem(g, O.dirs_for(wl.dirs), wl.bands)
    ost = p.init_state(g.T_init if T0 is None else T0)
    p.run(ost, wl.dt if dt is None else dt, wl.nsteps, wl.ninner, scheme)
    for which, key in ((bte.BTE_T_LATTICE, "TL"), (bte.BTE_T_PSEUDO, "Tp")):
        assert np.max(np.abs(s.T(0, which) - ost[key]) / ost[key]) <= 1e-12, key
    assert np.max(np.abs(s.intensity(0) - ost["I"]) / np.abs(ost["I"])) <= 1e-11


# bands (LA, TA, seed): 1 band (4 lanes a row), 9 (a padded row), 256 (the most)
@pytest.mark.parametrize("bands", [(1, 0, 51), (7, 2, 52), (240, 16, 53)])
@pytest.mark.parametrize("shape,dirs", [((3, 2, 1), W.Dirs("inplane", n_inplane=4)),
                                        ((1, 5, 1), W.Dirs("polar_azim", n_polar=4, n_azim=12)),
                                        ((3, 2, 2), W.Dirs("polar_azim", n_polar=2, n_azim=4))])
def test_rough_wall_ghosts(shape, dirs, bands):
    """Diffuse and partially specular sides on both ends of every axis."""
    dim = 2 if shape[2] == 1 else 3
    kinds = [W.BC_ISOTHERMAL, W.BC_DIFFUSE, W.BC_PARTIAL, W.BC_DIFFUSE, W.BC_DIFFUSE, W.BC_PARTIAL][:2 * dim]
    wl = workload(shape, dirs, bands, kinds, [308.0, 0.0, 0.35, 0.0, 0.0, 0.8][:2 * dim])
    s = bte.Solver(wl)
    s.step()
    check(wl, s)
    s.close()


# One block of rows (4 or 8 directions), several, and many; single cells, rows
# shorter and longer than a CTA's run of cells; band counts as above.
SHAPES = [((1, 1, 1), W.Dirs("inplane", n_inplane=4)), ((21, 3, 1), W.Dirs("inplane", n_inplane=12)),
          ((5, 4, 1), W.Dirs("polar_azim", n_polar=2, n_azim=4)), ((19, 2, 1), W.Dirs("polar_azim", n_polar=6, n_azim=12)),
          ((3, 2, 4), W.Dirs("inplane", n_inplane=8)), ((2, 17, 3), W.Dirs("polar_azim", n_polar=4, n_azim=8))]
ROWS = [({}, bte.BTE_IMPLICIT_JACOBI, 1), ({}, bte.BTE_IMPLICIT_JACOBI, 3),
        ({"fp64_strict": True}, bte.BTE_IMPLICIT_JACOBI, 3), ({"beta_exp": -1.2}, bte.BTE_IMPLICIT_JACOBI, 3),
        ({"beta_exp": 0.8}, bte.BTE_IMPLICIT_JACOBI, 1), ({}, bte.BTE_EXPLICIT, 1), ({"beta_exp": -0.7}, bte.BTE_EXPLICIT, 1)]


@pytest.mark.parametrize("kw,scheme,ninner", ROWS)
@pytest.mark.parametrize("shape,dirs", SHAPES)
def test_fp64_row_sweeps(shape, dirs, kw, scheme, ninner):
    """Every FP64 form of the row sweep, isothermal and mirror walls, from a
    non-uniform start."""
    dim = 2 if shape[2] == 1 else 3
    kinds = [W.BC_ISOTHERMAL, W.BC_SPECULAR, W.BC_SPECULAR, W.BC_ISOTHERMAL, W.BC_SPECULAR, W.BC_ISOTHERMAL][:2 * dim]
    explicit = scheme == bte.BTE_EXPLICIT
    wl = workload(shape, dirs, (9, 4, 54), kinds, [312.0, 0.0, 0.0, 304.0, 0.0, 299.0][:2 * dim],
                  dt=2e-13 if explicit else 1e-12, nsteps=3, ninner=ninner)
    T0 = W.random_temperatures(wl.geoms[0].ncells, 55, 296.0, 308.0)
    s = bte.Solver(wl, T_init=[T0], **kw)
    s.step(scheme=scheme)
    g = wl.geoms[0]
    p = O.Problem(g, O.dirs_for(wl.dirs), wl.bands, beta_exp=kw.get("beta_exp", 0.0))
    ost = p.init_state(T0)
    p.run(ost, wl.dt, wl.nsteps, wl.ninner, O.EXPLICIT if explicit else O.IMPLICIT)
    for which, key in ((bte.BTE_T_LATTICE, "TL"), (bte.BTE_T_PSEUDO, "Tp")):
        assert np.max(np.abs(s.T(0, which) - ost[key]) / ost[key]) <= 1e-12, key
    assert np.max(np.abs(s.intensity(0) - ost["I"]) / np.abs(ost["I"])) <= 1e-11
    s.close()


@pytest.mark.parametrize("bands", [(1, 0, 56), (240, 16, 57)])
@pytest.mark.parametrize("shape,dirs", [SHAPES[1], SHAPES[4], SHAPES[5]])
def test_fp64_row_sweep_band_counts(shape, dirs, bands):
    dim = 2 if shape[2] == 1 else 3
    wl = workload(shape, dirs, bands, [W.BC_ISOTHERMAL] * (2 * dim), [312.0, 300.0, 301.0, 304.0, 300.0, 299.0][:2 * dim])
    s = bte.Solver(wl)
    s.step()
    check(wl, s)
    s.close()


# FP32 storage: the reduced modes' bar, 1e-4 K; every team count of the tuner is timed and one kept
@pytest.mark.parametrize("tuned", [False, True])
@pytest.mark.parametrize("kw,scheme", [({}, bte.BTE_IMPLICIT_JACOBI), ({"beta_exp": -1.2}, bte.BTE_IMPLICIT_JACOBI),
                                       ({}, bte.BTE_EXPLICIT)])
@pytest.mark.parametrize("shape,dirs", SHAPES)
def test_fp32_row_sweeps(shape, dirs, kw, scheme, tuned):
    dim = 2 if shape[2] == 1 else 3
    kinds = [W.BC_ISOTHERMAL, W.BC_PARTIAL, W.BC_SPECULAR, W.BC_DIFFUSE, W.BC_SPECULAR, W.BC_ISOTHERMAL][:2 * dim]
    explicit = scheme == bte.BTE_EXPLICIT
    wl = workload(shape, dirs, (9, 4, 58), kinds, [309.0, 0.3, 0.0, 0.0, 0.0, 299.0][:2 * dim],
                  dt=2e-13 if explicit else 1e-12, nsteps=3, ninner=3)
    s = bte.Solver(wl, precision=bte.BTE_FP32, autotune=tuned, **kw)
    s.step(scheme=scheme)
    g = wl.geoms[0]
    p = O.Problem(g, O.dirs_for(wl.dirs), wl.bands, beta_exp=kw.get("beta_exp", 0.0))
    ost = p.init_state(g.T_init)
    p.run(ost, wl.dt, wl.nsteps, wl.ninner, O.EXPLICIT if explicit else O.IMPLICIT)
    for which, key in ((bte.BTE_T_LATTICE, "TL"), (bte.BTE_T_PSEUDO, "Tp")):
        assert np.max(np.abs(s.T(0, which) - ost[key])) <= 1e-4, key
    s.close()


@pytest.mark.parametrize("precision", [bte.BTE_FP64, bte.BTE_FP32, bte.BTE_BF16])
@pytest.mark.parametrize("dirs", [W.Dirs("inplane", n_inplane=12), W.Dirs("polar_azim", n_polar=4, n_azim=8)])
def test_intensities_keep_the_callers_direction_order(dirs, precision):
    """A state written and read back, and the direction table: the internal row
    order does not show."""
    wl = workload((4, 3, 1), dirs, (5, 2, 59), [W.BC_ISOTHERMAL] * 4, [305.0, 300.0, 300.0, 300.0])
    s = bte.Solver(wl, precision=precision)
    S, w, refl = bte.bte_get_directions(s.h)
    S_ref, w_ref, _ = O.dirs_for(wl.dirs)
    assert np.allclose(S, S_ref, rtol=1e-13, atol=1e-15) and np.allclose(w, w_ref, rtol=1e-13)
    for ax in range(3):
        M = S.copy()
        M[:, ax] *= -1
        assert np.allclose(S[refl[ax]], M, atol=1e-15)
    rng = np.random.default_rng(3)
    I0 = s.intensity(0)
    I = I0 * rng.uniform(0.99, 1.01, I0.shape)
    bte.bte_set_intensity(s.h, 0, I, np.full(12, 300.0))
    tol = {bte.BTE_FP64: 1e-14, bte.BTE_FP32: 1e-8, bte.BTE_BF16: 1e-4}[precision]   # 1 % deviations in 24 or 8 bits
    assert np.max(np.abs(s.intensity(0) - I) / I) <= tol
    s.close()


# 1024 cells is the last grid whose cell step is launched behind the running sweep; a
# random start queues every cell for the exact solve, a uniform one the few at the hot wall
@pytest.mark.parametrize("uniform", [False, True])
@pytest.mark.parametrize("shape", [(1, 1, 1), (32, 32, 1), (41, 25, 1)])
def test_cell_step_launches_and_queues(shape, uniform):
    wl = workload(shape, W.Dirs("inplane", n_inplane=4), (3, 1, 60), [W.BC_ISOTHERMAL] * 4, [330.0, 300.0, 300.0, 300.0],
                  nsteps=3)
    T0 = None if uniform else W.random_temperatures(wl.geoms[0].ncells, 61, 280.0, 320.0)
    s = bte.Solver(wl, **({} if uniform else {"T_init": [T0]}))
    s.step()
    check(wl, s, T0=T0)
    s.close()


# one pair of bands, a second pass of 64 bands, the most bands; runs of unequal weights
@pytest.mark.parametrize("bands", [(1, 0, 62), (50, 15, 63), (240, 16, 64)])
@pytest.mark.parametrize("kw", [{}, {"fp64_strict": True}])
def test_restored_energies(bands, kw):
    """T_L after a restore, from the sums formed while packing, against the T_L that the
    step's own sums gave for the same state."""
    wl = workload((3, 2, 1), W.Dirs("polar_azim", n_polar=6, n_azim=4), bands, [W.BC_ISOTHERMAL] * 4,
                  [310.0, 300.0, 303.0, 300.0])
    s = bte.Solver(wl, **kw)
    s.step()
    TL, I, Tp = s.T(0, bte.BTE_T_LATTICE), s.intensity(0), s.T(0, bte.BTE_T_PSEUDO)
    r = bte.Solver(wl, **kw)
    bte.bte_set_intensity(r.h, 0, I, Tp)
    assert np.max(np.abs(r.T(0, bte.BTE_T_LATTICE) - TL) / TL) <= 1e-12
    assert np.max(np.abs(r.intensity(0) - I) / I) <= 1e-14
    s.close()
    r.close()
