"""Rounding of the double-float sweep where it does not average out."""
import numpy as np
import pytest

from oracle import oracle as O
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


# One sweep of a uniform equilibrium changes nothing but by rounding.  I^n and the products
# with it are the same for all directions, so the mean over directions shows whether their
# rounding is too: 1.45e-15 rms over bands where I^n/(v dt) is formed first, 7.3e-16 where R I^n
# (R differs by direction) is, emulated.  Bar: 1.03e-15, half-way in the logarithm.  The intensities
# are given with 44 bits, which a pair of floats holds exactly.
def test_update_of_an_equilibrium():
    g = W.Geometry(2, 3, 3, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_SPECULAR] * 4, [0.0] * 4)
    bands = W.make_bands(40, 15, 85, log10_tau_range=(-9.0, -8.0))
    wl = W.Workload("equilibrium", [g], W.Dirs("polar_azim", n_polar=20, n_azim=20), bands, 2e-13, 1, 1)
    means = []
    for T in (270.0, 300.0, 330.0, 400.0, 450.0, 600.0):
        s = bte.Solver(wl, T_init=[np.full(9, T)])
        m, e = np.frexp(s.intensity(0))
        I = np.ldexp(np.round(m * 2.0**44), e - 44)
        bte.bte_set_intensity(s.h, 0, I, np.full(9, T))
        s.step()
        means.append(((s.intensity(0) - I) / I).mean(axis=1)[4])
        s.close()
    assert np.sqrt(np.mean(np.square(means))) <= 1.03e-15


# 1000 steps of 4 iterations of the same: the coefficients add up to one closely enough for the
# state to settle (1e-14 rms); with rounding errors of 2^-48 in their sum it drifts on (1.2e-13
# and more).  Bar: 3.5e-14, half-way in the logarithm.
def test_equilibrium_stays():
    g = W.Geometry(2, 4, 4, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_SPECULAR] * 4, [0.0] * 4)
    wl = W.Workload("equilibrium", [g], W.Dirs("polar_azim", n_polar=20, n_azim=20),
                    W.make_bands(40, 15, 85, log10_tau_range=(-6.0, -5.9)), 2e-13, 1, 1)
    s = bte.Solver(wl, use_graph=True)
    I0 = s.intensity(0)
    s.step(nsteps=1000, ninner=4)
    assert np.sqrt(np.mean(((s.intensity(0) - I0) / I0) ** 2)) <= 3.5e-14
    s.close()


# Steps so long that the coefficient W of I^n is 1e-6 to 1e-5, one cell at 300 K among cells and
# walls at 2 K, no scattering to speak of: where every upwind value is cold, the hot cell is left
# with W I^n alone.  W as 1 - R (...) would be off by 2^-49 / W, 3e-10 of it.  Bar: the FP64 parity bar
# on I.
def test_small_invariant_coefficient():
    g = W.Geometry(2, 2, 2, 1, 10e-9, 10e-9, 10e-9)
    W.uniform_walls(g, [W.BC_ISOTHERMAL] * 4, [2.0] * 4)
    bands = W.make_bands(8, 0, 86, log10_tau_range=(-3.0, -2.9))
    T0 = np.array([300.0, 2.0, 2.0, 2.0])
    for dt in (1e-6, 1e-7):
        wl = W.Workload("long step", [g], W.Dirs("polar_azim", n_polar=2, n_azim=4), bands, dt, 1, 1)
        s = bte.Solver(wl, T_init=[T0])
        s.step()
        p = O.Problem(g, O.dirs_for(wl.dirs), bands)
        ost = p.init_state(T0)
        p.run(ost, dt, 1, 1)
        I, ref = s.intensity(0), ost["I"]
        ok = ref > 1e-20  # below 2^-74 a pair keeps a float's bits
        assert ok.mean() > 0.3
        assert np.max(np.abs(I[ok] - ref[ok]) / ref[ok]) <= 1e-11
        s.close()
