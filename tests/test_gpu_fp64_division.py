"""The FP64 step divides by the density as IEEE does: Phi = rho u^3 with u = j / rho
comes back bit for bit as correctly rounded operations give it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g_mode_level", [0, 1])
def test_velocity_is_momentum_times_the_rounded_reciprocal(gpu_lib, g_mode_level):
    """d_0 and d_1 alone are given (d = f - w rho0, rho0 = 1), so that j_x = d_1 and
    rho = 1 + (d_0 + d_1) have one rounding each; densities from 1e-3 to 1e3.  With a
    periodic lattice's scalar and (level 1) vector kernel."""
    from paper_2312_10318_gb300 import Lattice
    n = 512
    rng = np.random.default_rng(5)
    f = np.empty((9, n, n))
    w = np.array([4.0 / 9] + [1.0 / 9] * 4 + [1.0 / 36] * 4)
    f[:] = w[:, None, None]
    f[0] = w[0] + (10.0 ** rng.uniform(-3, 3, (n, n)) - 1.0)
    f[1] = w[1] + rng.uniform(-0.1, 0.1, (n, n))
    lat = Lattice(n, n, 0.8, tau_s2=0.9, storage="f64")
    lat.set_kernel("vector" if g_mode_level else "scalar")
    lat.set_f(f, np.zeros((2, n, n))).step(1)
    phi = lat.get_f(with_phi=True)[1][0]
    d0, d1 = f[0] - w[0], f[1] - w[1]
    rho = 1.0 + ((d0 + 0.0) + (d1 + 0.0))
    ux = d1 * (1.0 / rho)
    assert np.array_equal(phi, ((rho * ux) * ux) * ux)
