"""Wall fluxes of rough walls, whatever form the state is held in: right after
bte_set_initial and after steps under other wall kinds, through both entry
points, against the FP64 oracle.  Bar: 1e-10 of the largest flux, as in the flux tests after steps
(an equilibrium state has none in its cells, only at its isothermal walls)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_19400_gb300 import bte, workloads as W

pytestmark = pytest.mark.gpu


def make(dim, kinds, temps):
    g = W.Geometry(dim, 5, 4, 1 if dim == 2 else 3, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, kinds, temps)
    return W.Workload("rough flux", [g], W.Dirs("polar_azim", n_polar=4, n_azim=8), W.make_bands(7, 3, 71), 1e-12, 2, 3)


def check(s, wl, I):
    """Both wall-flux calls (the one that allocates nothing first: it must not
    rely on the other's) and the cell fluxes against the oracle's of I."""
    g = wl.geoms[0]
    q_ref, qw_ref = O.Problem(g, O.dirs_for(wl.dirs), wl.bands).flux(I)
    scale = max(np.max(np.abs(q_ref)), np.max(np.abs(qw_ref)))
    qn = np.zeros(2 * g.dim)
    bte.bte_get_wall_flux_noalloc(s.h, 0, qn)
    q, qw = s.flux(0)
    assert np.max(np.abs(q - q_ref)) <= 1e-10 * scale
    assert np.max(np.abs(qw - qw_ref)) <= 1e-10 * scale
    assert np.array_equal(qn, qw)


SIDES = [(W.BC_DIFFUSE, 0.0), (W.BC_PARTIAL, 0.35)]


@pytest.mark.parametrize("kind,p", SIDES)
@pytest.mark.parametrize("dim", [2, 3])
def test_before_the_first_step(dim, kind, p):
    wl = make(dim, [W.BC_ISOTHERMAL, kind] * dim, [306.0, p] * dim)
    T0 = W.random_temperatures(wl.geoms[0].ncells, 72, 290.0, 315.0)
    s = bte.Solver(wl, T_init=[T0])
    check(s, wl, O.Problem(wl.geoms[0], O.dirs_for(wl.dirs), wl.bands).init_state(T0)["I"])
    s.close()


@pytest.mark.parametrize("kind,p", SIDES)
@pytest.mark.parametrize("dim", [2, 3])
def test_after_a_change_of_wall_kind(dim, kind, p):
    wl = make(dim, [W.BC_ISOTHERMAL, W.BC_SPECULAR] * dim, [306.0, 0.0] * dim)
    s = bte.Solver(wl)
    s.step()
    prob = O.Problem(wl.geoms[0], O.dirs_for(wl.dirs), wl.bands)
    ost = prob.init_state(wl.geoms[0].T_init)
    prob.run(ost, wl.dt, wl.nsteps, wl.ninner)
    for side in range(1, 2 * dim, 2):
        if kind == W.BC_PARTIAL:
            assert bte.lib().bte_set_specularity(s.h, 0, side, p) == bte.BTE_OK
        else:
            bte.bte_set_bc(s.h, 0, side, kind)
    rough = make(dim, [W.BC_ISOTHERMAL, kind] * dim, [306.0, p] * dim)
    check(s, rough, ost["I"])
    s.step(nsteps=1)  # and the state is the one the next step starts from
    O.Problem(rough.geoms[0], O.dirs_for(wl.dirs), wl.bands).run(ost, wl.dt, 1, wl.ninner)
    assert np.max(np.abs(s.T(0) - ost["TL"]) / ost["TL"]) <= 1e-12
    s.close()


# No heat crosses a wall at the temperature of a uniform state.  What is left is rounding: of the
# 252 partial sums 2e-17 of the one-sided flux, where one rounding error of the direction weights' sum,
# common to all bands, would leave 2.8e-16 on the x sides.  Bar: half of that.
def test_no_flux_at_equilibrium():
    g = W.Geometry(2, 3, 3, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_ISOTHERMAL] * 4, [300.0] * 4)
    wl = W.Workload("equilibrium", [g], W.Dirs("polar_azim", n_polar=20, n_azim=20), W.make_bands(40, 15, 72), 1e-12, 1, 1)
    s = bte.Solver(wl)
    S = bte.bte_get_directions(s.h)[0]
    one_sided = np.sum(s.intensity(0)[0] * np.maximum(S[:, :1], 0.0))
    q, qw = s.flux(0)
    assert np.max(np.abs(qw)) <= 1.4e-16 * one_sided
    s.close()
