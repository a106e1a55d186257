"""Grids whose beams end inside a warp, a block or an angle row: problems of a few beams, one row, rows
shorter than a warp and longer than a block, sizes around the launch shape's steps (128 beams a block,
one block an SM).  A few steps from a coherent state against the oracle, every integrator; and a batch
small enough for static slices beside one that takes pieces from the device-wide counter.

Tolerances: FP64 1e-11 (the sums' order and FMA contraction, a few roundings of 1e-16 a step, times the
largest phase a step turns, below 1e2); mixed 2e-6 (a few FP32 roundings of a unit state a step, ten
steps at most)."""
import numpy as np
import pytest

from bulb_inputs import Workload, coherent_unit_states
from oracle.integrate import dp45_step, evolve_adaptive, evolve_fixed, evolve_lie_adaptive
from oracle.physics import Bulb
from parity_util import beams, make_solver

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (1, 70), (63, 1), (64, 1), (65, 2), (31, 33), (300, 3), (127, 77), (33, 300)]
TOL = {"fp64": 1e-11, "mixed": 2e-6}


def state(wl, seed):
    psi = coherent_unit_states(wl.n_flavor, wl.n_beams, seed).reshape(2, wl.n_angle, wl.n_energy, wl.n_flavor)
    return psi[..., :, None] * np.conj(psi[..., None, :])


def oracle(wl, Y, h):
    b = Bulb(wl)
    r1 = wl.r0 + 2.5 * h
    if wl.integrator == "dp45":
        return evolve_adaptive(b, Y, wl.r0, r1, wl.rtol, wl.atol, h, h_max=h)[0]
    if wl.integrator == "lie_adaptive":
        return evolve_lie_adaptive(b, Y, wl.r0, r1, wl.rtol, wl.atol, h, h_max=h)[0]
    return evolve_fixed(b, Y, wl.r0, r1, 3, wl.integrator)[0]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nf,integrator", [(2, "rk4"), (2, "dp45"), (2, "lie_rk4"), (2, "lie_adaptive"), (3, "rk4"), (3, "dp45"),
                                           (3, "lie_rk4"), (3, "lie_adaptive")])
def test_edges(xf, nf, integrator, precision):
    for ne, nu in SIZES if nf == 2 else SIZES[:6]:
        wl = Workload(name="edge", n_flavor=nf, n_energy=ne, n_angle=nu, integrator=integrator, precision=precision,
                      dm2=(-2.4e-3, 0.0) if nf == 2 else (7.5e-5, -2.4e-3), theta=(0.1, 0, 0) if nf == 2 else (0.59, 0.15, 0.785),
                      matter="power_law", rtol=1e-4, atol=1e-4, r0=60.0)
        h = 2e-5                                           # turns the fastest beam by about 0.2
        Y = state(wl, seed=ne + nu)
        s = make_solver(xf, wl, h0_km=h, h_max_km=h, fixed_dr_km=2.5 * h / 3)
        s.set_rho(beams(Y), wl.r0)
        Y = s.get_rho().reshape(Y.shape)
        s.evolve(wl.r0, wl.r0 + 2.5 * h)
        got, st = s.get_rho(), s.stats()
        s.close()
        assert (st.accepted, st.rejected) == (3, 0)
        ref = beams(oracle(wl, Y, h))
        err = np.abs(got - ref).max()
        assert np.abs(ref - beams(Y)).max() > 1e-3         # the states moved
        assert err < TOL[precision], (ne, nu, err)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sizes", [[(17, 3), (64, 40), (5, 200)], [(50, 700), (33, 1500), (210, 1200), (128, 1900), (301, 1000), (400, 1333)]])
def test_batches_in_static_slices_and_in_pieces(xf, sizes, precision):
    h = 1e-3
    wls = [Workload(name=f"b{i}", n_energy=ne, n_angle=nu, integrator="dp45", precision=precision, rtol=1e-6, atol=1e-6, r0=100.0,
                    theta=(0.05 + 0.02 * i, 0, 0)) for i, (ne, nu) in enumerate(sizes)]
    s = xf.Solver([xf.config_from_workload(w, h0_km=h, h_max_km=h) for w in wls])
    for i, w in enumerate(wls):
        s.set_spectra(w.spectra(), inst=i)
    s.reset(100.0)
    s.evolve_batch(np.full(len(wls), 100.0 + 2.5 * h))
    for i, w in enumerate(wls):
        one = make_solver(xf, w, h0_km=h, h_max_km=h)
        one.reset(100.0)
        one.evolve(100.0, 100.0 + 2.5 * h)
        diff = np.abs(s.get_rho(xf.LAYOUT_NATIVE, inst=i) - one.get_rho(xf.LAYOUT_NATIVE)).max()
        assert diff < (1e-12 if precision == "fp64" else 1e-6), (sizes[i], diff)
        one.close()
    s.close()


@pytest.mark.parametrize("delta", [1.0, 1e-5, 1e-6])
def test_error_maximum_of_nearly_unpolarised_states(xf, delta):
    """The FP32 estimate that spares most beams the FP64 error norm must not pass over the largest
    ratio: states delta away from 1/3, whose norms are differences of nearly equal numbers, with a
    purely relative tolerance.  last_err against the oracle's; the FP64 rounding of the embedded error
    (1e-15 of a unit state) is below 1e-9 / delta of it, the error being above 1e-6 delta."""
    h = 1e-3
    wl = Workload(name="mix", n_flavor=3, n_energy=40, n_angle=90, integrator="dp45", precision="fp64", dm2=(7.5e-5, -2.4e-3),
                  theta=(0.59, 0.15, 0.785), matter="constant", lambda_const=1e3, rtol=1e-2, atol=0.0, r0=50.0)
    Y = np.eye(3) / 3 + delta * (state(wl, seed=5) - np.eye(3) / 3)
    s = make_solver(xf, wl, h0_km=h, h_max_km=h)
    s.set_rho(beams(Y), wl.r0)
    Y = s.get_rho().reshape(Y.shape)
    s.evolve(wl.r0, wl.r0 + h)
    st = s.stats()
    s.close()
    b = Bulb(wl)
    h = (wl.r0 + h) - wl.r0
    err = dp45_step(b.rhs, wl.r0, Y, h, b.rhs(wl.r0, Y), wl.atol, wl.rtol)[1]
    assert (st.accepted, st.rejected) == (1, 0) and err > 1e-4
    assert abs(st.last_err / err - 1) < 1e-9 / delta
