"""A masked lattice restored from get_f's populations and Phi advances two steps per
launch again, with the bits of single steps."""
import numpy as np
import pytest

from paper_2312_10318_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("first", [4, 5])
def test_restored_masked_lattices_keep_two_steps(gpu_lib, storage, first):
    from paper_2312_10318_gb300 import Lattice
    nx, ny = 80, 40
    mask = W.random_mask(nx, ny, seed=5, solid_frac=0.05, inlet_outlet=True, outlet=W.OUTLET)
    rho, ux, uy = W.random_fields(nx, ny, seed=9, u_amp=0.05, rho_amp=0.01)
    make = lambda: Lattice(nx, ny, 0.72, tau_s2=1.15, periodic=(False, True), wall_u=(0.03, 0.0), storage=storage,
                           mask=mask).set_two_step(True)
    run = make().init(ux, uy, rho).step(first)
    f, phi = run.get_f(with_phi=True)
    one, two = [make().set_f(f, phi) for _ in range(2)]
    one.set_kernel("scalar")
    assert two.two_step()
    for n in (5, 6):
        one.step(n)
        two.step(n)
        (fa, pa), (fb, pb) = one.get_f(with_phi=True), two.get_f(with_phi=True)
        assert np.array_equal(fa, fb) and np.array_equal(pa, pb)
    # another Phi at the solid nodes leaves them to single steps, until both buffers agree again
    other = np.where(mask == W.SOLID, 1e-3, phi)
    assert not two.set_f(f, other).two_step()
    assert two.set_f(f, phi).two_step()
    assert not two.set_f(f, other).step(1).set_f(f, phi).two_step()
