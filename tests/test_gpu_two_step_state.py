"""Saved and restored states of lattices that advance two steps per launch."""
import numpy as np
import pytest

from paper_2312_10318_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _masked(storage="f32", nx=70, ny=24):
    from paper_2312_10318_gb300 import Lattice
    solid = np.zeros((ny, nx), np.uint8)
    solid[8:12, 20:24] = W.SOLID
    return Lattice(nx, ny, 0.72, tau_s2=1.15, storage=storage, mask=solid).set_two_step(True), solid


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("first", [3, 4])
def test_an_image_with_a_given_phi_goes_on_bit_for_bit(gpu_lib, storage, first):
    """A Phi given for solid nodes sits in one of the two Phi buffers, which single
    steps read in turn: the lattice that loads such an image goes on as the saved one."""
    saved, solid = _masked(storage)
    rho, ux, uy = W.random_fields(70, 24, seed=3)
    saved.init(ux, uy, rho)
    saved.set_f(saved.get_f(), np.full((2, 24, 70), 1e-3)).step(first)
    image = saved.save()
    saved.step(6)
    loaded, _ = _masked(storage)
    loaded.load(image).step(6)
    (fa, pa), (fb, pb) = saved.get_f(with_phi=True), loaded.get_f(with_phi=True)
    assert np.array_equal(fa, fb) and np.array_equal(pa, pb)
    # and an image without one leaves the handle to two steps per launch again
    plain, _ = _masked(storage)
    plain.init(ux, uy, rho).step(first)
    image = plain.save()
    loaded.load(image)
    assert loaded.two_step()
    assert np.array_equal(loaded.step(6).get_f(), plain.step(6).get_f())
