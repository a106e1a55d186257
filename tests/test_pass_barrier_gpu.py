"""The stage barriers' own clock.  A stage barrier (no last block, every block waits for the count) that waits for
one arrival too many gives up after the configured limit: the step in flight is not taken, and the handle and
the device work again afterwards.  The moment launch, which would run out first, is left out by continuing an
advance whose moments are in place; a refused target makes the next call set the barrier words up again."""
import time

import pytest

from bulb_inputs import Workload
from oracle.physics import Bulb
from parity_util import beams, make_solver, oracle_run, rel_err

pytestmark = pytest.mark.gpu


def test_stage_barrier_runs_out(xf):
    wl = Workload(name="pb", n_energy=64, n_angle=32, integrator="rk4", n_steps=8, r0=100.0, r1=100.5)
    s = make_solver(xf, wl, barrier_timeout_ns=50_000_000)
    s.reset(100.0)
    s.advance([100.5], max_steps=2)
    before = s.stats()
    assert before.accepted == 2 and before.grid_blocks > 1
    with pytest.raises(xf.XflatError) as e:
        s.advance([1.0], max_steps=1)
    assert e.value.code == xf.ERR_INVAL
    s.debug_barrier_extra(1)
    t0 = time.perf_counter()
    s.advance(None, max_steps=2)
    after = s.stats()                            # synchronises
    assert 0.05 <= time.perf_counter() - t0 < 2.0
    assert after.accepted == 2 and after.r_km == before.r_km
    s.debug_barrier_extra(0)
    s.reset(100.0)
    s.evolve(100.0, 100.5)
    Y, _ = oracle_run(wl, Bulb(wl).initial_state(), 100.0, 100.5)
    assert rel_err(s.get_rho(), beams(Y)) < 1e-10
    s.close()
