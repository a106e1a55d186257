"""Dynamic piece scheduling (tests/dynamic_cases.py: the piece counter and its parity across passes and launches,
large and small pieces, pieces cut by the table's rows, stage states that one block writes and another reads):
through the bounds-checked build, against the instances alone, and under graph replay."""
import os
import subprocess
import sys

import numpy as np
import pytest

import dynamic_cases as dc

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
# three steps of short radial length: FP64 sums in another order and other contractions into FMAs; FP32 a few
# ulps (6e-8) a stage, about 20 stages
TOL = {"fp64": 1e-12, "mixed": 1e-5}


@pytest.fixture(scope="module")
def results(xf):
    return dc.run_cases(xf)


def test_bounds_checked_build(xf, results, tmp_path):
    from paper_1912_10596_gb300 import build
    build.build(variant="bounds")
    out = str(tmp_path / "dynamic.npz")
    res = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "dynamic_cases.py"), out], cwd=ROOT,
                         env=dict(os.environ, XFLAT_VARIANT="bounds"), capture_output=True, text=True, timeout=1200)
    report = res.stdout[-2000:] + res.stderr[-4000:]
    assert res.returncode == 0, report
    assert "dynamic cases ok" in res.stdout and "libxflat_bounds.so" in res.stdout, report
    got = np.load(out)
    assert sorted(got.files) == sorted(results)
    for k, ref in results.items():
        assert np.abs(got[k] - ref).max() <= TOL[k.split("_")[0]], k


@pytest.mark.parametrize("integrator,precision", dc.CASES)
def test_instances_alone(xf, results, integrator, precision):
    for i, wl in enumerate(dc.workloads(integrator, precision)):
        s = dc.batch(xf, [wl])
        s.evolve_batch(dc.target([wl]))
        diff = np.abs(s.get_rho(xf.LAYOUT_NATIVE) - results[f"{precision}_{integrator}{i}"]).max()
        assert diff <= TOL[precision], (i, diff)
        s.close()


@pytest.mark.parametrize("integrator,precision", [("dp45", "fp64"), ("lie_adaptive", "mixed"), ("dp45", "mixed")])
def test_graph_replay(xf, integrator, precision):
    wls = dc.workloads(integrator, precision)
    out = []
    for graph in (False, True):
        s = dc.batch(xf, wls)
        s.advance([dc.R0 + 40 * dc.H] * len(wls), max_steps=1)
        if graph:
            s.advance_graph(3, max_steps=2)
            s.advance_graph(3, max_steps=2)
        else:
            for _ in range(6):
                s.advance(None, max_steps=2)
        out.append([s.get_rho(xf.LAYOUT_NATIVE, inst=i) for i in range(len(wls))] + [s.stats(inst=i).accepted for i in range(len(wls))])
        s.close()
    assert out[0][len(wls):] == out[1][len(wls):] == [13] * len(wls)
    for a, b in zip(out[0][:len(wls)], out[1]):
        assert np.array_equal(a, b)
