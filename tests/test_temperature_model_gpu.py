"""Accuracy of the per-cell temperature model at the ends of its range."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_19400_gb300 import bte, mesh as M, workloads as W

pytestmark = pytest.mark.gpu


# The sums of the T_p equation scale with the relaxation rates: 1e14 1/s makes the
# model's slope about 1e20 (its square leaves the FP32 range), 1e-27 about 1e-21 (its
# square vanishes in FP32).  The walls move the wall cells' T_p by 1e-5 to 1e-4 of T, inside
# the model's trust radius.  Bar: the FP64 parity bar, T to rel 1e-12.
RATES = [(1e14, 301.0), (1e-27, 300.02)]


@pytest.mark.parametrize("beta,hot", RATES)
@pytest.mark.parametrize("scheme", [bte.BTE_IMPLICIT_JACOBI, bte.BTE_IMPLICIT_GS])
def test_model_root_does_not_depend_on_the_scale_of_the_rates(scheme, beta, hot):
    g = W.Geometry(2, 7, 5, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_ISOTHERMAL] * 4, [hot, 300.0, 300.0, 300.0])
    wl = W.Workload("rates", [g], W.Dirs("polar_azim", n_polar=2, n_azim=8), W.make_bands(9, 4, 75), 1e-12, 2, 3)
    wl.bands.beta = beta * wl.bands.beta / wl.bands.beta.max()
    s = bte.Solver(wl)
    s.step(scheme=scheme)
    p = O.Problem(g, O.dirs_for(wl.dirs), wl.bands)
    ost = p.init_state(300.0)
    p.run(ost, wl.dt, wl.nsteps, wl.ninner, O.GAUSS_SEIDEL if scheme == bte.BTE_IMPLICIT_GS else O.IMPLICIT)
    for which, key in ((bte.BTE_T_LATTICE, "TL"), (bte.BTE_T_PSEUDO, "Tp")):
        assert np.max(np.abs(s.T(0, which) - ost[key]) / ost[key]) <= 1e-12, key
    s.close()


@pytest.mark.parametrize("beta,hot", RATES)
def test_model_root_on_an_unstructured_mesh(beta, hot):
    m = M.tri_grid(5, 4, 50e-9, 40e-9, jitter=0.2, seed=76)
    bc = {t: (bte.BTE_BC_ISOTHERMAL, hot if t == 0 else 300.0) for t in m.tags}
    dirs, bands = W.Dirs("polar_azim", n_polar=2, n_azim=8), W.make_bands(9, 4, 75)
    bands.beta = beta * bands.beta / bands.beta.max()
    s = bte.UMeshSolver(m, dirs, bands, bc)
    s.step(1e-12, 2, 3)
    u = O.UMeshProblem(m, O.dirs_for(dirs), bands, bc)
    ost = u.init_state(300.0)
    u.run(ost, 1e-12, 2, 3)
    for which, key in ((bte.BTE_T_LATTICE, "TL"), (bte.BTE_T_PSEUDO, "Tp")):
        assert np.max(np.abs(s.T(which) - ost[key]) / ost[key]) <= 1e-12, key
    s.close()
