"""The two-step kernel's second buffers go back when an allocation needs them, also
those of a batch's members unless a captured run of the batch names them."""
import numpy as np
import pytest

from paper_2312_10318_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NX, NY = 2048, 1024          # second buffer 75 MB


def _members(stream, n=2):
    from paper_2312_10318_gb300 import Lattice
    _, ux, uy = W.random_fields(NX, NY, seed=8, u_amp=0.05, rho_amp=0.01)
    out = [Lattice(NX, NY, 0.7, tau_s2=0.9, storage="f32", stream=stream).init(ux, uy) for _ in range(n)]
    assert all(lat.two_step() for lat in out)
    return out


def _fill(leave_mib):
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - (leave_mib << 20), dtype=torch.uint8, device="cuda")


def _large(stream):
    """218 MB: 130 MiB and two second buffers, not one."""
    from paper_2312_10318_gb300 import Lattice
    return Lattice(2 * NX, NY, 0.7, tau_s2=0.9, storage="f32", stream=stream)


def _check(members, steps):
    import torch
    torch.cuda.empty_cache()
    ref = _members(members[0]._stream, 1)[0].set_kernel("scalar").step(steps)
    for lat in members:
        assert np.array_equal(lat.get_f(), ref.get_f())


def test_batches_without_captured_runs_leave_the_buffers_free_to_go(gpu_lib):
    import torch
    from paper_2312_10318_gb300.lattice import Batch
    stream = torch.cuda.Stream()
    for batch_stream, steps in ((stream, 5), (0, 40)):
        members = _members(batch_stream)
        batch = Batch(batch_stream).set(members).step(steps)
        filler = _fill(130)
        large = _large(stream)
        assert not any(lat.two_step() for lat in members)
        del filler
        large.close()
        batch.step(3)
        _check(members, steps + 3)
        batch.close()
        for lat in members:
            lat.close()


def test_a_batch_lets_go_with_its_captured_runs(gpu_lib):
    import torch
    from paper_2312_10318_gb300._lib import TrtrlbError
    from paper_2312_10318_gb300.lattice import Batch
    stream = torch.cuda.Stream()
    members = _members(stream)
    batch = Batch(stream).set(members).step(70)
    filler = _fill(130)
    with pytest.raises(TrtrlbError):
        _large(stream)
    assert all(lat.two_step() for lat in members)
    batch.step(70)                         # the captured run is still good
    batch.set(members)                     # and goes here
    large = _large(stream)
    assert not any(lat.two_step() for lat in members)
    del filler
    large.close()
    batch.step(7)
    _check(members, 147)
    batch.close()
    members = _members(stream)
    batch = Batch(stream).set(members).step(70)
    for lat in members:                    # before the batch, whose captured runs name their buffers
        lat.close()
    batch.close()
