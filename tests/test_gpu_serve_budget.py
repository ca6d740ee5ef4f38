"""The server's budget bounds what the admitted lattices occupy, second population
buffers included, and admits as many of them as fit without those buffers."""
import pytest

pytestmark = pytest.mark.gpu


def test_second_buffers_stay_within_the_budget_and_make_room(gpu_lib):
    from paper_2312_10318_gb300 import serve as S
    n, steps = 256, 200
    need = S.lattice_bytes(n, n, "f32")
    srv = S.Server(hbm_budget=4.5 * need, chunk=40)
    seen, step = [], srv.batch.step

    def watch(k):
        members = srv.batch.members
        seen.append((len(members), sum(L.device_bytes() for L in members), any(L.two_step() for L in members)))
        return step(k)

    srv.batch.step = watch
    reqs = [S.Request(k, "double_shear_layer", n, 1e4, steps, "f32") for k in range(6)]
    res = srv.run(reqs, realtime=False)
    assert [r.status for r in res] == ["ok"] * 6
    assert max(m for m, _, _ in seen) == 4
    # (4 KiB: the float of a lattice_bytes estimate against allocations)
    assert all(b <= srv.budget + 4096 for _, b, _ in seen)
    assert any(two for _, _, two in seen) and srv.used == 0 and srv.extra == 0
    # the results are those of a budget without limits
    free = S.Server(chunk=40)
    for a, b in zip(res, free.run(reqs, realtime=False)):
        assert a.diagnostics == b.diagnostics
