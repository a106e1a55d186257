"""The FP32 estimate that spares most beams the FP64 error norm, for states far below unit length: without
neutrino weights the equations are linear, and with a purely relative tolerance the error ratio does not
depend on the states' scale.  A factor 2^k is exact in double, so the largest ratio and the states agree
bit for bit.  The handles give every thread ten beams and more, as the estimate is first used for a thread's
second one."""
import numpy as np
import pytest

from bulb_inputs import Workload, random_unit_states

pytestmark = pytest.mark.gpu


def run(xf, wl, psi, k):
    n = wl.n_flavor
    s = xf.Solver(xf.config_from_workload(wl, h0_km=wl.h0, h_max_km=wl.h0, block_size=128, blocks_per_sm=1))
    s.set_spectra(np.zeros((2, n, wl.n_energy)))
    P = psi[:, :, None] * np.conj(psi[:, None, :])
    if n == 2:
        y = np.stack([2 * P[:, 0, 1].real, -2 * P[:, 0, 1].imag, (P[:, 0, 0] - P[:, 1, 1]).real])
    else:
        y = np.stack([P[:, 0, 0].real, P[:, 1, 1].real, P[:, 2, 2].real, P[:, 0, 1].real, P[:, 0, 1].imag, P[:, 0, 2].real,
                      P[:, 0, 2].imag, P[:, 1, 2].real, P[:, 1, 2].imag])
    s.set_rho(y * 2.0 ** k, wl.r0, layout=xf.LAYOUT_NATIVE)
    s.evolve(wl.r0, wl.r0 + wl.h0)
    st = s.stats()
    out = s.get_rho(xf.LAYOUT_NATIVE) * 2.0 ** -k
    s.close()
    return (st.accepted, st.rejected), st.last_err, out


@pytest.mark.parametrize("nf", [2, 3])
def test_error_maximum_does_not_depend_on_the_scale(xf, nf):
    wl = Workload(name="scale", n_flavor=nf, n_energy=200, n_angle=600, integrator="dp45", dm2=(-2.4e-3, 0.0) if nf == 2 else (7.5e-5, -2.4e-3),
                  theta=(0.4, 0, 0) if nf == 2 else (0.59, 0.15, 0.785), matter="constant", lambda_const=400.0, rtol=1e-4, atol=0.0,
                  h0=1e-3, r0=50.0)
    psi = random_unit_states(nf, wl.n_beams, 11)
    ref = run(xf, wl, psi, 0)
    assert ref[0] == (1, 0) and 1e-3 < ref[1] < 1.0
    for k in (-30, -55, -60, -63, -66, -72, -75, -100, -200, 60, 100):
        got = run(xf, wl, psi, k)
        assert got[0] == (1, 0) and got[1] == ref[1], (k, got[1], ref[1])
        assert np.array_equal(got[2], ref[2]), k
