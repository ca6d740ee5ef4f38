"""Runs of steps captured into a caller's CUDA graph: an even number of captured
steps returns to the buffers it began with, so every replay goes on from where
the one before ended, in every G mode, alone and in a batch, with and without
steps of its own in between."""
import numpy as np
import pytest

from paper_2312_10318_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _lattice(nx, ny, storage, g_mode, seed, stream, **kw):
    import torch
    from paper_2312_10318_gb300 import Lattice
    rho, ux, uy = W.random_fields(nx, ny, seed=seed, u_amp=0.05, rho_amp=0.01)
    lat = Lattice(nx, ny, 0.7, tau_s2=0.9, g=(2e-5, -1e-5), storage=storage, g_mode=g_mode, stream=stream, **kw)
    lat.init(ux, uy, rho)
    torch.cuda.synchronize()
    return lat


def _graph(step, n, stream):
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        step(n)
    return g


def _replay(g, stream):
    import torch
    with torch.cuda.stream(stream):
        g.replay()


def _same(a, b):
    (fa, pa), (fb, pb) = a.get_f(with_phi=True), b.get_f(with_phi=True)
    return np.array_equal(fa, fb) and np.array_equal(pa, pb)


@pytest.mark.parametrize("storage,g_mode,periodic", [("f32", "lagged", (True, True)), ("f32", "lagged", (True, False)),
                                                     ("f16", "lagged", (True, True)), ("bf16", "off", (False, True)),
                                                     ("f32", "current", (True, True)),
                                                     ("f16", "current", (True, True))])
@pytest.mark.parametrize("start", [0, 1])
def test_captured_even_runs_replay(gpu_lib, storage, g_mode, periodic, start):
    import torch
    stream = torch.cuda.Stream()
    for n in (2, 4, 6, 8, 64):
        one = _lattice(70, 33, storage, g_mode, n, stream, periodic=periodic).set_kernel("scalar")
        two = _lattice(70, 33, storage, g_mode, n, stream, periodic=periodic).set_two_step(True)
        assert two.two_step()
        one.step(start)
        two.step(start)
        g = _graph(two.step, n, stream)
        for k in range(3):
            _replay(g, stream)
            one.step(n)
            assert _same(one, two), (n, k)
        # steps of its own between replays, an even number in all
        two.step(3)
        two.step(1)
        _replay(g, stream)
        one.step(4 + n)
        assert _same(one, two), n


@pytest.mark.parametrize("n", [2, 6, 10])
def test_captured_batches_replay(gpu_lib, n):
    """Members of several formats and parities (classes beside one another)."""
    import torch
    from paper_2312_10318_gb300.lattice import Batch
    stream = torch.cuda.Stream()
    ones, twos = [], []
    for q, (st, g_mode, nx, ny) in enumerate([("f32", "lagged", 130, 40), ("f32", "lagged", 64, 33),
                                              ("f16", "current", 61, 40), ("f64", "lagged", 40, 20)]):
        for out in (ones, twos):
            lat = _lattice(nx, ny, st, g_mode, q, stream)
            if out is ones:
                lat.set_kernel("scalar")
            else:
                lat.set_two_step(True)
            out.append(lat.step(q % 2))
    batch = Batch(stream).set(twos)
    g = _graph(batch.step, n, stream)
    for _ in range(3):
        _replay(g, stream)
    batch.step(5)
    batch.step(1)
    _replay(g, stream)
    for q, (a, b) in enumerate(zip(ones, twos)):
        assert _same(a.step(4 * n + 6), b), q
