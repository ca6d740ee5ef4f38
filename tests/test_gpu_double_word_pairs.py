"""The double-word step with two nodes per thread in packed operations (periodic
lattices) gives the bits of the one with a node per thread, which a mask of fluid
nodes selects: heights with a row left over, narrow and wide tiles, both levels."""
import numpy as np
import pytest

from paper_2312_10318_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g_mode", ["lagged", "off"])
@pytest.mark.parametrize("nx,ny", [(1, 80001), (5, 16001), (90000, 1), (33, 2500), (130, 1033), (300, 331), (900, 901),
                                   (64, 1), (40, 3), (130, 33)])       # the last three: one node per thread too
def test_two_nodes_per_thread_give_the_bits_of_one(gpu_lib, nx, ny, g_mode):
    from paper_2312_10318_gb300 import Lattice
    rho, ux, uy = W.random_fields(nx, ny, seed=nx, u_amp=0.05, rho_amp=0.01)
    fluid = np.zeros((ny, nx), np.uint8)
    for g in ((2e-5, -1e-5), (0.0, 0.0)):
        two, one = [Lattice(nx, ny, 0.7, tau_s2=0.9, g=g, storage="f64dw", g_mode=g_mode, mask=m).init(ux, uy, rho)
                    for m in (None, fluid)]
        for n in (1, 4):
            (fa, pa), (fb, pb) = [lat.step(n).get_f(with_phi=True) for lat in (two, one)]
            assert np.array_equal(fa, fb) and np.array_equal(pa, pb), n
