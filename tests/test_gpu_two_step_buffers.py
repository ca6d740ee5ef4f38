"""How much memory the two-step kernel's second buffers may take, and giving one back."""
import numpy as np
import pytest

from paper_2312_10318_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_no_second_buffer_where_less_than_half_of_the_device_is_free(gpu_lib):
    import torch
    from paper_2312_10318_gb300 import Lattice
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    filler = torch.empty(free - total // 2 - (100 << 20), dtype=torch.uint8, device="cuda")
    lat = Lattice(2048, 1024, 0.7, tau_s2=0.9, storage="f32")     # 109 MB and a second buffer of 75
    assert not lat.two_step()
    del filler
    torch.cuda.empty_cache()
    assert Lattice(2048, 1024, 0.7, tau_s2=0.9, storage="f32").two_step()


@pytest.mark.parametrize("g_mode", ["lagged", "current"])
def test_two_steps_on_and_off(gpu_lib, g_mode):
    """Off gives the buffer back with the state in either of the two; with Phi at the
    current level, where both belong to single steps too, it can be put on again,
    beside a chosen single-step kernel."""
    from paper_2312_10318_gb300 import Lattice
    nx, ny = 130, 70
    rho, ux, uy = W.random_fields(nx, ny, seed=6, u_amp=0.05, rho_amp=0.01)
    for first in (2, 3, 5):
        a, b = [Lattice(nx, ny, 0.7, tau_s2=0.9, storage="f32", g_mode=g_mode).init(ux, uy, rho) for _ in range(2)]
        a.set_kernel("scalar").step(first + 9)
        held = b.step(first).device_bytes()
        b.set_two_step(False).step(4)
        assert not b.two_step()
        assert held - b.device_bytes() == (0 if g_mode == "current" else 36 * 192 * ny)
        b.set_kernel("column" if g_mode == "current" else "auto").set_two_step(True)
        assert b.two_step() == (g_mode == "current")
        b.step(5)
        assert np.array_equal(a.get_f(), b.get_f()), first
