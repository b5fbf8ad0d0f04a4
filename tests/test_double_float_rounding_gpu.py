"""Rounding of the double-float sweep where it does not average out."""
import numpy as np
import pytest

from paper_2305_19400_gb300 import bte, workloads as W

pytestmark = pytest.mark.gpu


# One band and a time step so short that every cell keeps its equilibrium: all directions of a
# cell have the same value, whose repeated addition is the worst case of an unnormalised pair
# (twenty in a row: 1.5e-14 rms relative, emulated; block by block: 2e-15).  E_L against the FP64
# sum of the intensities read back.  Bar: 6e-15 rms, half-way in the logarithm.
@pytest.mark.parametrize("dirs", [W.Dirs("inplane", n_inplane=20), W.Dirs("polar_azim", n_polar=20, n_azim=20),
                                  W.Dirs("polar_azim", n_polar=4, n_azim=40)])
def test_direction_sums_of_equal_values(dirs):
    g = W.Geometry(2, 30, 31, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_SPECULAR] * 4, [0.0] * 4)
    wl = W.Workload("sums", [g], dirs, W.make_bands(1, 0, 83), 1e-22, 1, 1)
    s = bte.Solver(wl, T_init=[W.random_temperatures(g.ncells, 84, 250.0, 500.0)])
    s.step()
    ref = np.einsum("pd,d->p", s.intensity(0)[:, :, 0], bte.bte_get_directions(s.h)[1]) / wl.bands.vg[0]
    err = (s.T(0, bte.BTE_E_LATTICE) - ref) / ref
    assert np.sqrt(np.mean(err ** 2)) <= 6e-15
    s.close()
