"""The mean survival probability over angle bins of one to a few warps of energies (the sums of several bins
share a warp up to 16 energies), against a plain FP64 sum over the state that the handle returns.  Both are
sums of non-negative terms: a few hundred roundings of 1.1e-16 at most, 1e-13."""
import numpy as np
import pytest

from bulb_inputs import Workload, random_unit_states
from parity_util import make_solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nf", [2, 3])
@pytest.mark.parametrize("ne", [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 64, 65])
def test_mean_survival(xf, ne, nf, precision):
    nu = 75                                                    # rows end inside a warp and a block
    wl = Workload(name="pee", n_flavor=nf, n_energy=ne, n_angle=nu, precision=precision,
                  dm2=(-2.4e-3, 0.0) if nf == 2 else (7.5e-5, -2.4e-3), theta=(0.1, 0, 0) if nf == 2 else (0.59, 0.15, 0.785))
    s = make_solver(xf, wl)
    psi = random_unit_states(nf, wl.n_beams, ne)
    s.set_rho(psi[:, :, None] * np.conj(psi[:, None, :]), 60.0)
    p = s.get_rho()[: nu * ne, 0, 0].real.reshape(nu, ne)
    N = wl.spectra()[0, 0]
    per_beam, mean = s.pee()
    _, alone = s.pee(per_beam=False)
    s.close()
    assert np.abs(per_beam[: nu * ne].reshape(nu, ne) - p).max() < 1e-15
    assert mean == alone == pytest.approx((N * p).sum() / (nu * N.sum()), rel=1e-13)
