"""The tuner and the two-step kernel: with Phi at the current level the 16-bit formats
get it where it is the faster one, and cached timings of older kernels are taken again."""
import json

import pytest

from paper_2312_10318_gb300 import tune as T

PER = (True, True)


class _Lattice:
    """Stands in for a Lattice in Tuner.apply."""

    def __init__(self, storage, g_mode, nx=512, ny=512):
        self.storage, self.g_mode, self.nx, self.ny = storage, g_mode, nx, ny
        self.calls = []

    def set_kernel(self, variant, tw):
        self.calls.append((variant, tw))

    def set_two_step(self, on):
        self.calls.append(on)


def _tuner(tmp_path, times):
    t = T.Tuner(cache_path=str(tmp_path / "tune.json"))
    t.runs = 0

    def measure(storage, nx, ny, periodic=PER, g_mode="lagged", **kw):
        t.runs += 1
        return dict(times)

    t.measure = measure
    return t


@pytest.mark.parametrize("two,faster", [(0.5, True), (2.0, False)])
def test_16_bit_current_phi_lattices_get_two_steps_where_faster(tmp_path, two, faster):
    t = _tuner(tmp_path, {"scalar:0": 1.5, "column:0": 1.0, "two_step": two})
    lat = _Lattice("f16", "current")
    assert t.apply(lat, PER) == ("column", 0)
    assert lat.calls == [("column", 0)] + [True] * faster
    again = _Lattice("f16", "current")           # from the cache, in another process too
    t2 = T.Tuner(cache_path=str(tmp_path / "tune.json"))
    t2.apply(again, PER)
    assert again.calls == lat.calls and not t2.measured


def test_cached_timings_of_other_kernels_are_taken_again(tmp_path):
    old = {"f32/periodic/current/512x512": {"variant": "column", "tile_w": 0, "ms_per_step": 1.0,
                                            "candidates": {"scalar:0": 3.0, "auto:0": 2.0, "column:0": 1.0}}}
    (tmp_path / "tune.json").write_text(json.dumps(old))
    t = _tuner(tmp_path, {"scalar:0": 3.0, "auto:0": 0.5, "column:0": 1.0})
    assert t.choose("f32", 512, 512, g_mode="current") == ("auto", 0) and t.runs == 1
    assert t.choose("f32", 512, 512, g_mode="current") == ("auto", 0) and t.runs == 1


@pytest.mark.gpu
def test_tuned_16_bit_current_phi_lattices(gpu_lib, tmp_path):
    import numpy as np
    from paper_2312_10318_gb300 import Lattice, workloads as W
    t = T.Tuner(cache_path=str(tmp_path / "tune.json"), steps=32, reps=2)
    pr = W.double_shear_layer(1024, re=1e4)
    a, b = [Lattice(1024, 1024, pr.tau_s, storage="f16", g_mode="current", **pr.lattice_kwargs()) for _ in range(2)]
    t.apply(a, pr.periodic)
    e = t.table["f16/periodic/current/1024x1024"]
    assert a.two_step() == (e["two_step_ms"] < e["ms_per_step"])
    b.set_kernel("scalar")
    for lat in (a, b):
        lat.init(pr.ux, pr.uy).step(7)
    assert np.array_equal(a.get_f(), b.get_f())
