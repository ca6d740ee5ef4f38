"""Handles on different threads: one changes kernels and steps while another thread's
allocation takes back the first one's second buffer."""
import threading

import numpy as np
import pytest

from paper_2312_10318_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_a_buffer_taken_back_by_another_thread(gpu_lib):
    import torch
    from paper_2312_10318_gb300 import Lattice
    nx, ny = 2048, 1024
    _, ux, uy = W.random_fields(nx, ny, seed=8, u_amp=0.05, rho_amp=0.01)
    for _ in range(4):
        one, two = [Lattice(nx, ny, 0.7, tau_s2=0.9, storage="f32", stream=torch.cuda.Stream()).init(ux, uy)
                    for _ in range(2)]
        one.set_kernel("scalar")
        assert two.two_step()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        filler = torch.empty(torch.cuda.mem_get_info()[0] - (130 << 20), dtype=torch.uint8, device="cuda")
        steps, begun, stop, errors = [0], threading.Event(), threading.Event(), []

        def run():
            try:
                while not stop.is_set() or steps[0] < 30:
                    two.set_kernel("scalar").set_kernel("auto").step(3)
                    steps[0] += 3
                    begun.set()
            except Exception as e:         # reported by the test's own thread
                errors.append(e)
                begun.set()

        t = threading.Thread(target=run)
        t.start()
        begun.wait()
        # 218 MB: the 130 left and both second buffers (75 each)
        other = Lattice(2 * nx, ny, 0.7, tau_s2=0.9, storage="f32", stream=torch.cuda.Stream())
        stop.set()
        t.join()
        assert not errors
        assert not one.two_step() and not two.two_step()
        del filler
        torch.cuda.empty_cache()
        one.step(steps[0])
        assert np.array_equal(one.get_f(), two.get_f())
        for lat in (one, two, other):
            lat.close()
