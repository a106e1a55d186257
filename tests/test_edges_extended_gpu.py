"""Grids whose beams end inside a warp, a block or an angle row, for the exponential midpoint rule and the
extended model (azimuthal bins): three steps from a near-electron state against the oracle.

Tolerances: FP64 1e-11 (the sums' order and FMA contraction, a few roundings of 1e-16 a step, times the
largest phase a step turns, below 1e2); mixed 2e-6 (a few FP32 roundings of a unit state a step)."""
import numpy as np
import pytest

from bulb_inputs import Workload
from oracle.extended import ExtendedBulb
from oracle.integrate import evolve_adaptive, evolve_em2, evolve_fixed
from oracle.physics import Bulb
from parity_util import beams, make_solver
from test_block_edges_gpu import SIZES, TOL, state

pytestmark = pytest.mark.gpu


def run(xf, b, wl, Y, evolve, n_phi):
    h = 2e-5
    s = make_solver(xf, wl, h0_km=h, h_max_km=h, fixed_dr_km=2.5 * h / 3, n_phi=n_phi)
    s.set_rho(beams(Y), wl.r0)
    Y = s.get_rho().reshape(Y.shape)
    s.evolve(wl.r0, wl.r0 + 2.5 * h)
    got, st = s.get_rho(), s.stats()
    s.close()
    assert (st.accepted, st.rejected) == (3, 0)
    if evolve is evolve_fixed:
        ref = evolve(b, Y, wl.r0, wl.r0 + 2.5 * h, 3, wl.integrator)[0]
    else:
        ref = evolve(b, Y, wl.r0, wl.r0 + 2.5 * h, wl.rtol, wl.atol, h, h_max=h)[0]
    err = np.abs(got - beams(ref)).max()
    assert np.abs(beams(ref) - beams(Y)).max() > 1e-3          # the states moved
    assert err < TOL[wl.precision], (wl.n_energy, wl.n_angle, err)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nf", [2, 3])
def test_midpoint_edges(xf, nf, precision):
    for ne, nu in SIZES[:6]:
        wl = Workload(name="edge", n_flavor=nf, n_energy=ne, n_angle=nu, integrator="exp_midpoint", precision=precision,
                      dm2=(-2.4e-3, 0.0) if nf == 2 else (7.5e-5, -2.4e-3), theta=(0.1, 0, 0) if nf == 2 else (0.59, 0.15, 0.785),
                      matter="power_law", rtol=1.0, atol=1.0, r0=60.0)
        run(xf, Bulb(wl), wl, state(wl, seed=ne + nu), evolve_em2, 0)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("integrator,evolve", [("rk4", evolve_fixed), ("dp45", evolve_adaptive), ("lie_rk4", evolve_fixed)])
@pytest.mark.parametrize("n_phi", [2, 5])
def test_extended_edges(xf, integrator, evolve, precision, n_phi):
    for ne, nu in [(1, 1), (1, 35), (63, 1), (65, 2), (31, 33)]:
        wl = Workload(name="edge", n_energy=ne, n_angle=nu, integrator=integrator, precision=precision, matter="power_law",
                      rtol=1e-4, atol=1e-4, r0=60.0)
        eb = ExtendedBulb(wl, n_phi)
        wide = Workload(name="s", n_energy=ne, n_angle=nu * n_phi)
        Y = state(wide, seed=ne + nu).reshape(2, nu, n_phi, ne, 2, 2)
        run(xf, eb, wl, Y, evolve, n_phi)
