"""Relaxation rates far from those at T_ref: beta_b (T_p / T_ref)^p with p at the
end of its range."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2305_19400_gb300 import bte, workloads as W

pytestmark = pytest.mark.gpu


# (T / T_ref)^-16 = 4e37 and 2e38: 1 + (s - 1) A_s, whose reciprocal scales every
# coefficient, on both sides of the FP32 range's end.  Bar: the FP64 parity bar.
@pytest.mark.parametrize("T", [4.45, 4.0])
@pytest.mark.parametrize("ninner", [1, 3])
def test_rates_beyond_the_float_range(T, ninner):
    g = W.Geometry(2, 5, 4, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_ISOTHERMAL, W.BC_ISOTHERMAL, W.BC_SPECULAR, W.BC_SPECULAR], [T * 1.01, T, 0.0, 0.0])
    wl = W.Workload("rates", [g], W.Dirs("polar_azim", n_polar=2, n_azim=8), W.make_bands(6, 2, 78, omega_max=2e12),
                    1e-9, 1, ninner)
    s = bte.Solver(wl, T_init=[np.full(20, T)], beta_exp=-16.0, T_ref=1000.0)
    s.step()
    p = O.Problem(g, O.dirs_for(wl.dirs), wl.bands, beta_exp=-16.0, beta_Tref=1000.0)
    ost = p.init_state(T)
    p.run(ost, wl.dt, wl.nsteps, wl.ninner)
    assert np.max(np.abs(s.intensity(0) - ost["I"]) / ost["I"]) <= 1e-11
    assert np.max(np.abs(s.T(0, bte.BTE_T_PSEUDO) - ost["Tp"]) / ost["Tp"]) <= 1e-12
    s.close()
