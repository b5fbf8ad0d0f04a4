"""The initial state of an FP64 handle is held in full double precision until a
double-float step: what is read back, and what an IEEE step starts from, does not
depend on fp64_strict."""
import numpy as np
import pytest

from paper_2305_19400_gb300 import bte, workloads as W

pytestmark = pytest.mark.gpu


def workload(ngeom=1):
    geoms = []
    for k in range(ngeom):
        g = W.Geometry(2, 6, 5 + k, 1, 10e-9, 10e-9, 10e-9)
        W.uniform_walls(g, [W.BC_ISOTHERMAL] * 2 + [W.BC_SPECULAR] * 2, [303.0, 300.0, 0.0, 0.0])
        geoms.append(g)
    return W.Workload("initial", geoms, W.Dirs("polar_azim", n_polar=4, n_azim=8), W.make_bands(9, 4, 73), 1e-12, 1, 2)


# 5 K: intensities of the upper bands lie far below 2^-74, where a pair of floats keeps 24 bits or none
@pytest.mark.parametrize("T", [5.0, 300.0, 900.0])
def test_read_back_bit_for_bit(T):
    wl = workload()
    a, b = bte.Solver(wl, T_init=[np.full(30, T)]), bte.Solver(wl, T_init=[np.full(30, T)], fp64_strict=True)
    assert np.array_equal(a.intensity(0), b.intensity(0))
    a.close()
    b.close()


def test_one_geometry_set_again_after_a_step():
    """The others keep their state; the one that is set again starts in doubles."""
    wl = workload(2)
    s, ref = bte.Solver(wl), bte.Solver(wl, fp64_strict=True)
    s.step()
    other = s.intensity(1)
    T = W.random_temperatures(30, 74, 280.0, 320.0)
    for h in (s.h, ref.h):
        bte.bte_set_initial(h, 0, T)
    assert np.array_equal(s.intensity(0), ref.intensity(0))
    assert np.array_equal(s.intensity(1), other)
    s.close()
    ref.close()


@pytest.mark.parametrize("scheme", [bte.BTE_IMPLICIT_JACOBI, bte.BTE_EXPLICIT, bte.BTE_IMPLICIT_GS])
def test_tuning_leaves_the_state(scheme):
    s = bte.Solver(workload())
    I = s.intensity(0)
    bte.bte_autotune(s.h, 1e-13, scheme)
    assert np.array_equal(s.intensity(0), I)
    s.close()


def test_beside_a_restored_geometry():
    """A restore of one geometry leaves the other's initial state in full precision."""
    wl = workload(2)
    s, ref = bte.Solver(wl), bte.Solver(wl, fp64_strict=True)
    I0, I1 = ref.intensity(0), ref.intensity(1)
    bte.bte_set_intensity(s.h, 0, I0 * 1.01, np.full(30, 301.0))
    assert np.array_equal(s.intensity(1), I1)
    assert np.array_equal(s.intensity(0), I0 * 1.01)
    s.close()
    ref.close()


@pytest.mark.parametrize("scheme", [bte.BTE_EXPLICIT, bte.BTE_IMPLICIT_GS])
def test_an_ieee_step_starts_from_doubles(scheme):
    """Bit for bit the step of a handle whose state was read, and so written in doubles, before."""
    a, b = bte.Solver(workload()), bte.Solver(workload())
    b.intensity(0)
    for s in (a, b):
        s.step(dt=1e-13, scheme=scheme)
    assert np.array_equal(a.intensity(0), b.intensity(0))
    a.close()
    b.close()


def test_a_lone_geometry_set_again():
    wl = workload()
    a, b = bte.Solver(wl), bte.Solver(wl)
    a.step()
    bte.bte_set_initial(a.h, 0, np.full(30, 310.0))
    bte.bte_set_initial(b.h, 0, np.full(30, 310.0))
    b.intensity(0)  # b from doubles: the double-float step converts them
    for s in (a, b):
        s.step()
    assert np.array_equal(a.intensity(0), b.intensity(0))
    a.close()
    b.close()
