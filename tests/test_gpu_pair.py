"""The two-step kernel against single steps: the same bits, for every format and
G mode it runs, at the edges of its strips (60 nodes) and lattices narrower than
one, even and odd widths (paired and elementwise rows at the wrap), heights of
one band and less, and step counts of every split; alone and in batches (direct
launches and replayed runs from both parities), and after its second buffer has
been given back."""
import numpy as np
import pytest

from paper_2312_10318_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(32, 1), (33, 2), (59, 3), (60, 5), (61, 130), (62, 4), (121, 9), (122, 257), (250, 246)]


def _lattices(nx, ny, storage, g_mode, seed, n=2, **kw):
    from paper_2312_10318_gb300 import Lattice
    rho, ux, uy = W.random_fields(nx, ny, seed=seed, u_amp=0.05, rho_amp=0.01)
    return [Lattice(nx, ny, 0.7, tau_s2=0.9, g=(2e-5, -1e-5), storage=storage, g_mode=g_mode, **kw)
            .init(ux, uy, rho) for _ in range(n)]


def _same(a, b):
    (fa, pa), (fb, pb) = a.get_f(with_phi=True), b.get_f(with_phi=True)
    return np.array_equal(fa, fb) and np.array_equal(pa, pb) and \
        all(np.array_equal(x, y) for x, y in zip(a.moments(), b.moments()))


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("g_mode", ["lagged", "off"])
def test_two_steps_equal_single_steps(gpu_lib, storage, g_mode):
    for k, (nx, ny) in enumerate(SIZES):
        a, b = _lattices(nx, ny, storage, g_mode, k)
        a.set_kernel("scalar")
        assert b.two_step() and not a.two_step()
        for n in (1, 2, 3, 6, 7):
            a.step(n)
            b.step(n)
            assert a.t == b.t and _same(a, b), (nx, ny, n)


def _masks(nx, ny, seed):
    """(mask or None, periodic, wall_u): walls, obstacles, inlet and both outlets,
    and an outlet ghost column inside, in the first column a strip stores."""
    out = [(None, (True, False), (0.0, 0.0)), (None, (False, True), (0.0, 0.0)), (None, (False, False), (0.0, 0.0)),
           (W.random_mask(nx, ny, seed=seed, solid_frac=0.1), (True, True), (0.0, 0.0))]
    for outlet in (W.OUTLET, W.PRESSURE):
        m = W.random_mask(nx, ny, seed=seed + 1, solid_frac=0.05, inlet_outlet=True, outlet=outlet)
        out.append((m, (False, seed % 2 == 0), (0.03, 0.004)))
    if ny > 10 and nx > 62:
        m = np.zeros((ny, nx), np.uint8)
        m[4:10, 60:62] = W.SOLID
        m[5:9, 60] = W.OUTLET
        out.append((m, (True, True), (0.0, 0.0)))
    return out


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("g_mode", ["lagged", "off"])
def test_two_steps_equal_single_steps_with_walls_and_masks(gpu_lib, storage, g_mode):
    """Bands of one part and of several (1500 rows), plain and special tiles, rows and
    columns past open edges."""
    for k, (nx, ny) in enumerate([(32, 1), (33, 5), (64, 33), (130, 70), (301, 66), (1300, 1500)]):
        for mask, periodic, wall_u in _masks(nx, ny, k)[:3 if ny > 1000 else None]:
            a, b = _lattices(nx, ny, storage, g_mode, k, mask=mask, periodic=periodic, wall_u=wall_u)
            a.set_kernel("scalar")
            assert b.two_step() and not a.two_step()
            for n in (1, 2, 3, 6):
                a.step(n)
                b.step(n)
                assert _same(a, b), (nx, ny, periodic, mask is not None, n)


def test_lattices_the_two_step_kernel_leaves_to_single_steps(gpu_lib):
    """Halo classes, an outlet ghost that emits to its far side, a Phi given for
    solid nodes; and the same states all the same."""
    nx, ny = 70, 12
    halo = np.zeros((ny, nx), np.uint8)
    halo[0] = 5
    ghost = np.zeros((ny, nx), np.uint8)
    ghost[3, 40] = W.OUTLET
    for m in (halo, ghost):
        a, b = _lattices(nx, ny, "f32", "lagged", 1, mask=m)
        a.set_kernel("scalar")
        assert not b.two_step()
        assert _same(a.step(5), b.step(5))
    solid = np.zeros((ny, nx), np.uint8)
    solid[4:6, 10:12] = W.SOLID
    a, b = _lattices(nx, ny, "f32", "lagged", 2, mask=solid)
    a.set_kernel("scalar")
    phi = np.full((2, ny, nx), 1e-4)
    f = a.get_f()
    for lat in (a, b):
        lat.set_f(f, phi)
    assert not b.two_step() and _same(a.step(6), b.step(6))


def test_two_steps_in_batches(gpu_lib):
    import torch
    from paper_2312_10318_gb300.lattice import Batch
    stream = torch.cuda.Stream()
    alone, members = [], []
    for q, (st, nx, ny) in enumerate([("f32", 130, 70), ("f32", 64, 33), ("f16", 61, 40), ("f64", 40, 20),
                                      ("bf16", 300, 9), ("f32", 200, 65), ("f32", 130, 40)]):
        a, b = _lattices(nx, ny, st, "lagged", q, stream=stream, periodic=(True, q != 6))
        a.set_kernel("scalar")
        for lat in (a, b):
            lat.step(q % 2)                    # members at both parities
        alone.append(a)
        members.append(b)
    for group in ([0, 2, 4], [0, 1, 2, 3, 4, 5, 6]):   # all even, then mixed
        batch = Batch(stream).set([members[k] for k in group])
        for n in (3, 32, 33, 70, 64, 1, 65):
            batch.step(n)
            for k in group:
                alone[k].step(n)
        torch.cuda.synchronize()
        for k in group:
            assert _same(alone[k], members[k]), (group, k)


def test_second_buffer_is_given_back_when_memory_runs_out(gpu_lib):
    import torch
    from paper_2312_10318_gb300 import Lattice
    a, b = _lattices(4096, 2048, "f32", "lagged", 3)
    assert a.two_step() and b.two_step()
    held = b.device_bytes()
    z = torch.zeros((2048, 4096), dtype=torch.float64, device="cuda")
    for lat in (a, b):
        lat.init(z + 0.03, z)
        lat.step(4)                             # odd-level launches: the state may sit in either buffer
    b.step(2)
    a.set_kernel("scalar").step(2)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    filler = torch.empty(free - (200 << 20), dtype=torch.uint8, device="cuda")
    c = Lattice(4096, 2048, 0.7, magic=0.25, storage="f32")    # 436 MB, of which 236 are missing
    assert not b.two_step() and b.device_bytes() < held and c.t == 0
    del filler
    torch.cuda.empty_cache()
    for lat in (a, b):
        lat.step(3)
    assert _same(a, b)


def test_many_narrow_lattices_share_launches(gpu_lib):
    """Lattices narrower than a tile (widths 1 to 33, tiles of the next power of
    two) and more of them than one launch holds (96), periodic and walled: each
    ends where it ends alone."""
    import torch
    from paper_2312_10318_gb300 import Lattice
    from paper_2312_10318_gb300.lattice import Batch
    stream = torch.cuda.Stream()
    widths = (1, 2, 3, 5, 8, 9, 16, 17, 31, 33)
    alone, members = [], []
    for q in range(100):
        nx, ny = widths[q % len(widths)], 1 + 7 * (q % 6)
        rho, ux, uy = W.random_fields(nx, ny, seed=q, u_amp=0.05, rho_amp=0.01)
        for out in (alone, members):
            out.append(Lattice(nx, ny, 0.8, magic=0.25, periodic=(True, False), g=(1e-5, 0.0), storage="f64",
                               stream=stream).init(ux, uy, rho))
    Batch(stream).set(members).step(35)
    for a in alone:
        a.step(35)
    torch.cuda.synchronize()
    for q, (a, b) in enumerate(zip(alone, members)):
        assert _same(a, b), q


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_two_current_phi_steps_equal_single_steps(gpu_lib, storage):
    """With Phi at the current level (56 nodes stored per strip): the same bits as
    the plain and the column kernel's single steps."""
    for k, (nx, ny) in enumerate([(32, 1), (33, 2), (55, 3), (56, 5), (57, 130), (58, 4), (113, 9), (250, 246)]):
        a, c, b = _lattices(nx, ny, storage, "current", k, n=3)
        a.set_kernel("scalar")
        c.set_kernel("column")
        assert b.two_step() and not a.two_step()
        for n in (1, 2, 3, 6):
            for lat in (a, b, c):
                lat.step(n)
            assert _same(a, b) and _same(c, b), (nx, ny, n)


@pytest.mark.parametrize("g_mode", ["lagged", "off"])
def test_double_word_two_nodes_per_thread(gpu_lib, g_mode):
    """The periodic double-word step's pairs of rows (heights with a row left over,
    narrow and wide tiles) against FP64 storage."""
    for nx, ny, kw in [(64, 1, {}), (5, 3, {}), (40, 3, {}), (130, 33, {}), (300, 131, {}), (900, 901, {})]:
        rho, ux, uy = W.random_fields(nx, ny, seed=nx, u_amp=0.05, rho_amp=0.01)
        from paper_2312_10318_gb300 import Lattice
        a, b = [Lattice(nx, ny, 0.7, tau_s2=0.9, g=(2e-5, -1e-5), storage=s, g_mode=g_mode, **kw)
                .init(ux, uy, rho).step(5) for s in ("f64", "f64dw")]
        fa, fb = a.get_f(), b.get_f()
        # 5 steps of the format's 2^-47 relative to the largest population
        assert np.abs(fa - fb).max() <= 1e-12 * np.abs(fa).max(), (nx, ny)
