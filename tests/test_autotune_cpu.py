"""The autotuner's candidates and cache key, with the timing replaced: the library's own launch shape is among
the candidates wherever they do not list it already, and a stored choice holds for one library and one model."""
import ctypes as C
import types

import pytest

from paper_1912_10596_gb300 import autotune

FP64, MIXED = 0, 1


class Config(C.Structure):
    _fields_ = [(n, C.c_uint32) for n in ("n_flavor", "precision", "integrator", "n_energy", "n_angle", "n_phi",
                                          "block_size", "blocks_per_sm")]


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    torch = pytest.importorskip("torch")
    xf = types.SimpleNamespace(MIXED=MIXED, xflat_config=Config, XflatError=RuntimeError, _LIB_PATH=str(tmp_path / "lib.so"))
    timed = []

    def fake_time(xf, torch, cfgs, spectra, r_end, steps, warmup):
        shape = (cfgs[0].block_size, cfgs[0].blocks_per_sm)
        timed.append(shape)
        return (1.0 if shape == xf.fastest else 2.0), 0

    monkeypatch.setattr(autotune, "_time", fake_time)
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "cache.json"))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda: "gpu")

    def tune(library, fastest, **cfg):
        (tmp_path / "lib.so.sha256").write_text(library)
        xf.fastest = fastest
        timed.clear()
        return autotune.tune(xf, [Config(n_energy=10, n_angle=10, **cfg)], [None], [1.0]), list(timed)

    return tune


@pytest.mark.parametrize("cfg", [dict(n_flavor=2, precision=FP64), dict(n_flavor=3, precision=FP64),
                                 dict(n_flavor=3, precision=MIXED), dict(n_flavor=2, precision=MIXED, n_phi=4)])
def test_library_shape_and_two_blocks_are_tried(tuner, cfg):
    best, timed = tuner("a", (0, 0), **cfg)
    assert best == (0, 0) and (256, 2) in timed


def test_choice_holds_for_one_library_and_model(tuner):
    bulb, ext = dict(n_flavor=2, precision=MIXED), dict(n_flavor=2, precision=MIXED, n_phi=4)
    assert tuner("a", (512, 1), **bulb)[0] == (512, 1)
    assert tuner("a", (256, 3), **bulb) == ((512, 1), [])              # stored
    assert tuner("a", (256, 3), **ext)[0] == (256, 3)
    assert tuner("b", (256, 2), **bulb)[0] == (256, 2)
