"""The Bloch rotation of the exponential integrators at any angle: one exponential-midpoint step in a constant
matter potential alone (unit path factor, no vacuum term, no neutrino weights) turns the transverse
components by exactly h lambda, up to angles whose square leaves the FP32 range.

Tolerances: FP64, a few roundings of the half-angle formula; mixed, the angle itself is an FP32 number
(two units in the last place of it) and the state holds a few FP32 roundings."""
import numpy as np
import pytest

from bulb_inputs import Workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,angle", [("fp64", 0.5), ("fp64", 2.0 ** 10), ("fp64", 2.0 ** 62), ("fp64", 2.0 ** 63),
                                             ("fp64", 2.0 ** 65), ("fp64", -(2.0 ** 70)), ("fp64", 2.0 ** 200),
                                             ("mixed", 0.5), ("mixed", 2.0 ** 6), ("mixed", 2.0 ** 20)])
def test_rotation_by_a_constant_potential(xf, precision, angle):
    wl = Workload(name="turn", n_energy=9, n_angle=5, dm2=(0.0, 0.0), integrator="exp_midpoint", precision=precision,
                  rtol=1e-6, atol=1e-6, matter="constant", lambda_const=angle)
    s = xf.Solver(xf.config_from_workload(wl, geometry="homogeneous", mu_const_kmi=0.0, h0_km=1.0))
    s.set_spectra(np.zeros((2, 2, 9)))
    y = np.zeros((3, wl.n_beams))
    y[0] = 1.0
    s.set_rho(y, 100.0, layout=xf.LAYOUT_NATIVE)
    s.evolve(100.0, 101.0)
    got, st = s.get_rho(xf.LAYOUT_NATIVE), s.stats()
    s.close()
    assert (st.accepted, st.rejected) == (1, 0)
    tol = 1e-14 if precision == "fp64" else 1e-6 + 2.4e-7 * abs(angle)
    assert np.abs(got[2]).max() == 0.0
    if tol < 1.0:
        assert np.abs(got[0] - np.cos(angle)).max() < tol and np.abs(got[1] - np.sin(angle)).max() < tol
    assert np.abs(np.hypot(got[0], got[1]) - 1.0).max() < min(tol, 1e-6)
