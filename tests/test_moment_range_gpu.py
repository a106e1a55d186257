"""FP64 moments over the whole range of the fixed-point accumulators: angle weights of any size up to the
accumulators' 2^63, a clear refusal beyond it, and handles cut into many thousands of pieces, whose partial
sums all add to the same words."""
import numpy as np
import pytest

from bulb_inputs import Workload
from oracle.physics import Grid
from parity_util import random_state, beams

pytestmark = pytest.mark.gpu


def solver(xf, wl, scale):
    g = Grid.from_workload(wl)
    s = xf.Solver(xf.config_from_workload(wl))
    s.set_spectra(g.N, g.u, g.du * scale)
    s.set_rho(beams(random_state(wl, 3)), 100.0)
    return s


@pytest.mark.parametrize("nf,integrator", [(2, "rk4"), (2, "dp45"), (2, "lie_adaptive"), (3, "dp45")])
def test_moments_scale_with_the_angle_weights(xf, nf, integrator):
    """The sums are linear in the angle weights, and a factor 2^k is exact in double.  What differs is what the
    accumulators leave out, in units of the total weight: every block's partial below 2^-64, and 2^-54 where a
    negative sum is turned to double (its words are those of 1 - |x|); J0 and a traceless diagonal are sums of
    two such moments, and two handles are compared."""
    wl = Workload(name="scale", n_flavor=nf, n_energy=37, n_angle=61, integrator=integrator, n_steps=4,
                  dm2=(-2.4e-3, 0.0) if nf == 2 else (7.5e-5, -2.4e-3), theta=(0.1, 0, 0) if nf == 2 else (0.59, 0.15, 0.785))
    s = solver(xf, wl, 1.0)
    ref = np.stack(s.moments())
    blocks = s.stats().grid_blocks
    s.close()
    bound = 4 * np.abs(Grid.from_workload(wl).N).sum() * (2.0 ** -54 + blocks * 2.0 ** -64)
    assert bound < 1e-13 * np.abs(ref).max()
    for k in (1, 4, 10, 30, 50, 52, 55, 60):
        s = solver(xf, wl, 2.0 ** k)
        got = np.stack(s.moments()) / 2.0 ** k
        s.close()
        assert np.abs(got - ref).max() <= bound, k


@pytest.mark.parametrize("nf,integrator", [(2, "rk4"), (2, "dp45"), (2, "lie_adaptive"), (3, "dp45")])
def test_moments_beyond_the_accumulators_are_refused(xf, nf, integrator):
    """A sum of 2^63 and more does not fit; it is reported, not returned as some other number."""
    wl = Workload(name="beyond", n_flavor=nf, n_energy=37, n_angle=61, integrator=integrator, n_steps=4,
                  dm2=(-2.4e-3, 0.0) if nf == 2 else (7.5e-5, -2.4e-3), theta=(0.1, 0, 0) if nf == 2 else (0.59, 0.15, 0.785))
    for k in (80, 200):
        s = solver(xf, wl, 2.0 ** k)
        with pytest.raises(xf.XflatError) as e:
            s.moments()
        assert e.value.code == xf.ERR_NONFINITE, k
        s.close()


@pytest.mark.parametrize("n_angle", [300_000, 1_000_000])
def test_moments_of_many_pieces(xf, n_angle):
    """One energy bin: a piece holds at most 128 angle rows, so these handles have 4,700 and 16,000 pieces
    with partial sums of the same sign.  Pure flavour states: J1 = N_e / 2 sigma_z and J0 the same times the
    mean of 1/cos.  Tolerance: FP64 sums of 1e6 equal terms in runs of 128, a few 1e-14."""
    wl = Workload(name="pieces", n_energy=1, n_angle=n_angle, integrator="lie_rk4", n_steps=1)
    s = xf.Solver(xf.config_from_workload(wl))
    N = np.zeros((2, 2, 1))
    N[0, 0] = 1.0
    s.set_spectra(N)
    s.reset(100.0)
    J0, J1 = s.moments()
    s.close()
    u = (np.arange(n_angle) + 0.5) / n_angle
    q = (1.0 / np.sqrt(1.0 - u * (wl.R_km / 100.0) ** 2)).mean()
    assert abs(J1[0, 0] - 0.5) < 1e-13 and abs(J1[1, 1] + 0.5) < 1e-13
    assert abs(J0[0, 0] - 0.5 * q) < 1e-13 and abs(J0[1, 1] + 0.5 * q) < 1e-13
