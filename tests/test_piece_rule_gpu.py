"""Which batches take their pieces from the device-wide counter: below ten vector iterations a block, mixed
two-flavour handles whose static slices would hold four pieces and more (angle rows of few energies), and
no others.  The results are those of the instances alone (mixed sums are exact: 1e-6 for the FP32
roundings of the moments over three steps; FP64 1e-12, another order of the sums)."""
import numpy as np
import pytest

from bulb_inputs import Workload
from dynamic_cases import H, R0, takes_pieces

pytestmark = pytest.mark.gpu

SHORT = [(16, 3600), (301, 300), (23, 3000), (20, 900)]      # up to five pieces of 47 rows in a block's share
LONG = [(300, 200), (301, 300), (333, 200), (150, 120)]


def make(xf, sizes, integrator, precision):
    s = xf.Solver([xf.config_from_workload(Workload(name="p", n_energy=e, n_angle=u, integrator=integrator, precision=precision,
                                                    rtol=1e-4, atol=1e-4, r0=R0), h0_km=H, h_max_km=H) for e, u in sizes])
    for i, (e, u) in enumerate(sizes):
        s.set_spectra(Workload(name="p", n_energy=e, n_angle=u).spectra(), inst=i)
    s.reset(R0)
    return s


@pytest.mark.parametrize("sizes,integrator,precision,pieces", [(SHORT, "dp45", "mixed", True), (SHORT, "lie_adaptive", "mixed", True),
                                                               (LONG, "dp45", "mixed", False), (SHORT, "dp45", "fp64", False)])
def test_pieces_or_slices(xf, sizes, integrator, precision, pieces):
    r1 = np.full(len(sizes), R0 + 2.5 * H)
    s = make(xf, sizes, integrator, precision)
    assert takes_pieces(xf, s, lambda: s.evolve_batch(r1)) == pieces
    for i, size in enumerate(sizes):
        one = make(xf, [size], integrator, precision)
        one.evolve_batch(r1[:1])
        diff = np.abs(s.get_rho(xf.LAYOUT_NATIVE, inst=i) - one.get_rho(xf.LAYOUT_NATIVE)).max()
        assert diff < (1e-12 if precision == "fp64" else 1e-6), (size, diff)
        one.close()
    s.close()
