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
