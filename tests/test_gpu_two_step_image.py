"""Images of equal runs are equal byte for byte, whatever the device memory held
before the lattice was made."""
import numpy as np
import pytest

from paper_2312_10318_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("masked", [False, True])
def test_images_of_equal_runs_are_equal(gpu_lib, storage, masked):
    """Before each run, lattices of the same allocation sizes without padding columns
    (128 wide, the run's 100 have 28) leave their values in the memory that the
    run's lattice then gets."""
    from paper_2312_10318_gb300 import Lattice
    ny = 16
    mask = None
    if masked:
        mask = np.zeros((ny, 100), np.uint8)
        mask[5:9, 40:50] = W.SOLID
    rho, ux, uy = W.random_fields(100, ny, seed=4, u_amp=0.05, rho_amp=0.01)
    images = []
    for seed in (11, 12):
        r, u, v = W.random_fields(128, ny, seed=seed, u_amp=0.05, rho_amp=0.01)
        old = [Lattice(128, ny, 0.7, tau_s2=0.9, storage=storage).init(u, v, r).step(5) for _ in range(40)]
        for lat in old:
            lat.diagnostics()
        for lat in old[1::2]:                  # the others keep the blocks they share
            lat.close()
        lat = Lattice(100, ny, 0.7, tau_s2=0.9, storage=storage, mask=mask).init(ux, uy, rho).set_two_step(True)
        assert lat.two_step()
        images.append(lat.step(3).save())      # one launch of two steps: the second buffer
        lat.close()
    assert np.array_equal(*images)
