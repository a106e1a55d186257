"""The three-flavour propagator exp(-i Om) rho exp(i Om) (Eq. U for 3 x 3 generators) over the sizes and
shapes of Om where its closed form could go wrong: zero, far below and far above one radian, two
nearly equal eigenvalues (matter far above the vacuum splittings), diagonal.

One Lie RK4 step with a constant generator (no nu-nu term to speak of, constant matter, radial beams
of the single-angle geometry) is exactly that propagator, so the step is compared with a 64-bit
eigen-decomposition of the same generator.
"""
import numpy as np
import pytest

from bulb_inputs import Workload
from oracle.physics import e_projector, vacuum_hamiltonian
from parity_util import random_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("mixing", [(0.59, 0.15, 0.785), (0.0, 0.0, 0.0)])
@pytest.mark.parametrize("lam,h", [(0.0, 0.0), (0.0, 1e-9), (0.0, 0.5), (1e-6, 1e-3), (1.0, 1.0), (1e3, 1e-2),
                                   (1e5, 1e-2), (1e5, 1e-12)])
def test_constant_generator(xf, precision, mixing, lam, h):
    ne, nu, r0 = 37, 5, 50.0
    # h = 0: the smallest splittings and step stand in for Om = 0 (a step has a length)
    dm2 = (7.5e-5, 2.4e-3) if h else (1e-300, 1e-300)
    h = h or 1e-9
    wl = Workload(name="prop", n_flavor=3, n_energy=ne, n_angle=nu, integrator="lie_rk4", precision=precision, dm2=dm2,
                  theta=mixing, matter="constant", lambda_const=lam, n_steps=1, r0=r0, r1=r0 + h)
    s = xf.Solver(xf.config_from_workload(wl, geometry="single_angle", fixed_dr_km=h))
    s.set_spectra(np.ones((2, 3, ne)) * np.array([1.0, 1.0, 1.0])[None, :, None])      # N_e = N_x: no nu-nu term
    Y = random_state(wl, seed=3).reshape(-1, 3, 3)
    s.set_rho(Y, r0)
    Y = s.get_rho()                                                                    # as the handle holds it
    s.evolve(r0, r0 + h)
    got = s.get_rho()
    s.close()
    h = (r0 + h) - r0                                                                  # the step that was taken
    E = 1.0 + (np.arange(ne) + 0.5) * (60.0 - 1.0) / ne
    H = vacuum_hamiltonian(E, 3, dm2, mixing)
    gen = np.stack([H + lam * e_projector(3), H - lam * e_projector(3)])[:, None]      # nu, nubar (paper's own Pbar)
    l, V = np.linalg.eigh(np.broadcast_to(gen, (2, nu, ne, 3, 3)).reshape(-1, 3, 3))
    U = (V * np.exp(-1j * h * l)[:, None, :]) @ np.conj(np.swapaxes(V, 1, 2))
    ref = U @ Y @ np.conj(np.swapaxes(U, 1, 2))
    # two propagators of 16 roundings each, the generator's entries and phases to a few more, and in
    # mixed precision the purification: 64 roundings of max(1, |Om|)
    norm = h * float(np.abs(gen).max()) * 3.0
    eps = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    assert np.abs(got - ref).max() <= 64 * eps * max(1.0, norm)
