"""The adjoint kernel where a block holds many beams and angle rows, against the oracle's discrete adjoint: a
thread walks several rows (sums flushed between them), the partials of all blocks are summed in strides, and,
with more than 64 rows a block, the row values are computed a beam at a time instead of tabulated.

Tolerance: a few hundred roundings of 1.1e-16 in the states and again in their adjoints, of order one against
luminosity gradients of about 0.05: below 1e-11 of the largest; 1e-10."""
import numpy as np
import pytest

from bulb_inputs import Workload
from oracle.adjoint import rk4_adjoint
from oracle.physics import Bulb

pytestmark = pytest.mark.gpu
L = {"nue": 4e51, "nuebar": 3e51, "nux": 1e51, "nuxbar": 1e51}


@pytest.mark.parametrize("ne,nu,steps", [(13, 3001, 16),      # 40 rows a block, about two beams a thread
                                         (7, 6001, 16),       # 79 rows a block
                                         (2, 6000, 24)])      # 79 rows a block, less than a beam a thread
def test_many_rows_a_block(xf, ne, nu, steps):
    wl = Workload(name="rows", n_energy=ne, n_angle=nu, integrator="rk4", n_steps=steps, dm2=(2.4e-3, 0.0), theta=(0.2, 0.0, 0.0),
                  matter="constant", lambda_const=3.0, L=L)
    b = Bulb(wl)
    Jo, GNo, Gtho = rk4_adjoint(b, b.initial_state(), 100.0, 101.0, steps)
    s = xf.Solver(xf.config_from_workload(wl))
    s.set_spectra(b.grid.N)
    J, dN, dth = s.adjoint(100.0, 101.0, steps, 5)
    s.close()
    assert J == pytest.approx(Jo, rel=1e-12)
    scale = np.abs(GNo * b.grid.N).max()
    assert scale > 0.01
    assert np.abs((dN - GNo) * b.grid.N).max() < 1e-10 * scale
    assert dth == pytest.approx(Gtho, rel=1e-10)
