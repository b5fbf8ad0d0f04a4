"""E_L after a restore: the sum of the restored values in double precision, for any
values and whatever T_p comes with them."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_19400_gb300 import bte, mesh as M, workloads as W

pytestmark = pytest.mark.gpu

DIRS, BANDS = W.Dirs("polar_azim", n_polar=4, n_azim=8), W.make_bands(40, 15, 79)


def energy(I, w):
    return np.einsum("pdb,d,b->p", I, w, 1.0 / BANDS.vg)


# 32 directions x 55 bands of the same sign: a few ulp in any order of FP64 addition;
# the bar leaves room for 100.  scale: intensities that have nothing to do with I0(T_p).
@pytest.mark.parametrize("precision", [bte.BTE_FP64, bte.BTE_FP32, bte.BTE_BF16])
@pytest.mark.parametrize("scale", [1.0, 1e-9])
def test_structured(precision, scale):
    g = W.Geometry(2, 3, 2, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_ISOTHERMAL] * 4, [300.0] * 4)
    s = bte.Solver(W.Workload("restore", [g], DIRS, BANDS, 1e-12, 1, 1), precision=precision)
    rng = np.random.default_rng(80)
    I = s.intensity(0) * scale * rng.uniform(0.9, 1.1, (6, 32, 55))
    bte.bte_set_intensity(s.h, 0, I, np.full(6, 300.0))
    ref = energy(s.intensity(0), bte.bte_get_directions(s.h)[1])
    floor = energy(I / scale, bte.bte_get_directions(s.h)[1]) if precision != bte.BTE_FP64 else ref  # deviations are stored
    assert np.max(np.abs(s.T(0, bte.BTE_E_LATTICE) - ref) / floor) <= 2e-14
    s.close()


# T_L of the restored energies (E_L itself is not read from this handle): the FP64 parity bar
@pytest.mark.parametrize("scale", [1.0, 1e-6])
def test_unstructured(scale):
    m = M.tri_grid(3, 2, 30e-9, 20e-9, jitter=0.2, seed=81)
    bc = {t: (bte.BTE_BC_ISOTHERMAL, 300.0) for t in m.tags}
    s = bte.UMeshSolver(m, DIRS, BANDS, bc)
    rng = np.random.default_rng(82)
    I = s.intensity() * scale * rng.uniform(0.9, 1.1, (m.ncells, 32, 55))
    s.set_state(I, np.full(m.ncells, 300.0))
    w = O.dirs_for(DIRS)[1]
    p = O.UMeshProblem(m, O.dirs_for(DIRS), BANDS, bc).tables
    ref = np.array([p.solve_T(np.sum(w) / BANDS.vg, E, 100.0)[0] for E in energy(I, w)])
    assert np.max(np.abs(s.T(bte.BTE_T_LATTICE) - ref) / ref) <= 1e-12
    s.close()
