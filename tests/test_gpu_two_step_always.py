"""The two-step kernels on lattices of every size, where runs would take single steps
because these are faster: the comparisons of test_gpu_pair.py with
set_two_step(True), and what a run of small lattices takes by itself."""
import numpy as np
import pytest

import test_gpu_pair as pair

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def always(monkeypatch):
    made = pair._lattices
    monkeypatch.setattr(pair, "_lattices",
                        lambda *a, **kw: [lat.set_two_step(True) for lat in made(*a, **kw)])


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("g_mode", ["lagged", "off"])
def test_periodic(gpu_lib, storage, g_mode):
    pair.test_two_steps_equal_single_steps(gpu_lib, storage, g_mode)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("g_mode", ["lagged", "off"])
def test_walls_and_masks(gpu_lib, storage, g_mode):
    pair.test_two_steps_equal_single_steps_with_walls_and_masks(gpu_lib, storage, g_mode)


def test_batches(gpu_lib):
    pair.test_two_steps_in_batches(gpu_lib)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_current_phi(gpu_lib, storage):
    pair.test_two_current_phi_steps_equal_single_steps(gpu_lib, storage)


def test_what_runs_take_by_themselves(gpu_lib):
    """The rule's inputs from the lattices: alone, in a batch, replayed or not; and the
    same bits whichever way the run goes."""
    import torch
    from paper_2312_10318_gb300 import Lattice, workloads as W
    from paper_2312_10318_gb300.lattice import Batch
    stream = torch.cuda.Stream()
    make = lambda nx, ny, **kw: Lattice(nx, ny, 0.8, tau_s2=1.0, stream=stream, **kw)
    wall, cur = make(64, 64, periodic=(True, False)), make(64, 64, g_mode="current")
    assert wall.two_step() and not wall.two_step_run() and wall.set_two_step(True).two_step_run()
    assert make(66, 64).two_step_run() and Batch(stream).set([make(66, 64)]).two_step_run()
    assert cur.two_step_run() and not Batch(stream).set([cur]).two_step_run()
    curs = [make(64, 64, g_mode="current") for _ in range(20)]
    assert Batch(stream).set(curs).two_step_run()
    assert not make(64, 64, storage="f64").two_step_run()
    # replayed single steps and a rest of launches of two
    rho, ux, uy = W.random_fields(64, 40, seed=2, u_amp=0.05, rho_amp=0.01)
    ref, a = [make(64, 40, g_mode="current").init(ux, uy, rho) for _ in range(2)]
    ref.set_kernel("scalar")
    batch = Batch(stream).set([a])
    for n in (63, 32, 70):
        batch.step(n)
        assert np.array_equal(ref.step(n).get_f(), a.get_f())
    # one member on, the other by the rule: they go the way of the run together
    rho, ux, uy = W.random_fields(64, 40, seed=2, u_amp=0.05, rho_amp=0.01)
    ref, a, b = [make(64, 40, periodic=(True, False)).init(ux, uy, rho) for _ in range(3)]
    a.set_two_step(True)
    batch = Batch(stream).set([a, b])
    for n in (3, 70, 32):
        batch.step(n)
        ref.step(n)
        torch.cuda.synchronize()
        assert np.array_equal(ref.get_f(), a.get_f()) and np.array_equal(ref.get_f(), b.get_f())
