"""Temperature solves where hbar omega >> k_B T."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_19400_gb300 import bte, workloads as W

pytestmark = pytest.mark.gpu

RTOL = 1e-14  # the default newton_rtol


# One band at the top of the range, x = hbar omega / (k_B T) = 150 to 380, started a
# relative distance q from the root: an accepted step's error is the remainder of a
# Taylor model, in T about x^(n-1) q^n / n! for one that leaves out the term of order n.
# Bar: that of the model of second order at its radius (rtol / 4)^(1/3), x^2 rtol / 24,
# which the model of third order must not exceed, plus rounding.
@pytest.mark.parametrize("T", [2.0, 3.0, 5.0])
@pytest.mark.parametrize("q", [8e-5, 1.25e-4, -1.25e-4])
def test_solve_of_a_high_band(T, q):
    g = W.Geometry(2, 2, 2, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_ISOTHERMAL] * 4, [300.0] * 4)
    bands = W.Bands(np.array([9.9e13]), np.array([1e14]), np.array([5e3]), np.array([1e11]), np.array([1.0]))
    wl = W.Workload("band", [g], W.Dirs("inplane", n_inplane=4), bands, 1e-12, 1, 1)
    s = bte.Solver(wl)
    Wtot = float(np.sum(bte.bte_get_directions(s.h)[1]))
    Ep = Wtot * O.I0(bands, T)[0][0] * bands.beta[0] / bands.vg[0]
    got, _ = bte.bte_solve_T(s.h, np.array([Ep]), T0=np.array([T * (1.0 + q)]))
    x = 1.054571817e-34 * 1e14 / (1.380649e-23 * T)
    assert abs(got[0] - T) / T <= x * x * RTOL / 24.0 + 1e-14
    s.close()


# Whole steps at 4 to 30 K.  Bar: the FP64 parity bar on T.
@pytest.mark.parametrize("T", [4.0, 12.0, 30.0])
@pytest.mark.parametrize("kw", [{}, {"fp64_strict": True}])
def test_steps_at_low_temperature(T, kw):
    g = W.Geometry(2, 6, 4, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_ISOTHERMAL, W.BC_ISOTHERMAL, W.BC_SPECULAR, W.BC_SPECULAR], [T * 1.002, T, 0.0, 0.0])
    wl = W.Workload("cold", [g], W.Dirs("polar_azim", n_polar=2, n_azim=8), W.make_bands(40, 15, 77), 1e-12, 2, 4)
    s = bte.Solver(wl, T_init=[np.full(24, T)], **kw)
    s.step()
    p = O.Problem(g, O.dirs_for(wl.dirs), wl.bands)
    ost = p.init_state(T)
    p.run(ost, wl.dt, wl.nsteps, wl.ninner)
    for which, key in ((bte.BTE_T_LATTICE, "TL"), (bte.BTE_T_PSEUDO, "Tp")):
        assert np.max(np.abs(s.T(0, which) - ost[key]) / ost[key]) <= 1e-12, key
    s.close()
