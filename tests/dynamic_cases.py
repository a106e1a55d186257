"""Batches large enough that their blocks take pieces from the device-wide counter (ten vector iterations of
a block), through the library the binding loads (XFLAT_VARIANT selects a checking build): FP64 with stored
stage derivatives, and the adaptive exact propagators, whose stage states wait in the output planes, in FP64
and mixed precision.  `run_cases()` returns the final states by case name, after making sure from the pass
trace that the handle took the dynamic path; as a script it writes them to an .npz file."""
import ctypes as C
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))
sys.path.insert(0, HERE)

from bulb_inputs import Workload  # noqa: E402

# uneven sizes, one with rows so short that the table's rows cut its pieces; 128 threads on one block an SM
SIZES = {"fp64": [(100, 501), (33, 801), (64, 377), (5, 3001)], "mixed": [(101, 1001), (33, 1601), (64, 755), (5, 6001)]}
SHAPE = dict(block_size=128, blocks_per_sm=1)
CASES = [("dp45", "fp64"), ("rk4", "fp64"), ("lie_adaptive", "fp64"), ("lie_adaptive", "mixed"), ("dp45", "mixed")]
H, R0, STEPS = 1e-3, 100.0, 3


def workloads(integrator, precision):
    return [Workload(name=f"d{i}", n_energy=ne, n_angle=nu, integrator=integrator, precision=precision, rtol=1e-5, atol=1e-5, r0=R0,
                     theta=(0.05 + 0.02 * i, 0, 0)) for i, (ne, nu) in enumerate(SIZES[precision])]


def config(xf, wl):
    return xf.config_from_workload(wl, h0_km=H, h_max_km=H, fixed_dr_km=H, **SHAPE)


def target(wls):
    return np.full(len(wls), R0 + (STEPS - (0.0 if wls[0].integrator == "rk4" else 0.5)) * H)


def batch(xf, wls):
    s = xf.Solver([config(xf, w) for w in wls])
    for i, w in enumerate(wls):
        s.set_spectra(w.spectra(), inst=i)
    s.reset(R0)
    return s


def takes_pieces(xf, s, advance):
    """Whether the stage passes of the next launch end in a barrier with a last block, as only those of
    handles with dynamic pieces do (xflat_debug_trace)."""
    grid = C.c_uint32(0)
    assert xf.xflat_debug_trace(s.h, 1, None, C.byref(grid)) == xf.OK
    advance()
    t = np.zeros((1, grid.value, 4), dtype=np.uint64)
    assert xf.xflat_debug_trace(s.h, 1, t.ctypes.data_as(C.c_void_p), None) == xf.OK
    assert xf.xflat_debug_trace(s.h, 0, None, None) == xf.OK
    assert (t[0, :, 0] != 0).all()
    return bool((t[0, :, 3] != 0).any())


def run_cases(xf):
    out = {}
    for integrator, precision in CASES:
        wls = workloads(integrator, precision)
        s = batch(xf, wls)
        assert takes_pieces(xf, s, lambda: s.evolve_batch(target(wls))), (integrator, precision)
        for i in range(len(wls)):
            out[f"{precision}_{integrator}{i}"] = s.get_rho(xf.LAYOUT_NATIVE, inst=i)
        s.close()
    return out


if __name__ == "__main__":
    from paper_1912_10596_gb300 import xflat
    res = run_cases(xflat)
    np.savez(sys.argv[1], **res)
    print(f"dynamic cases ok {len(res)} {os.path.basename(xflat._LIB_PATH)}")
