"""When a run takes two steps per launch: the rule on sizes (csrc/lb_pair_rule.h),
compiled and called on the host, at shapes on both sides of its lines."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include <cstdio>
#include <cstdlib>
#include "lb_pair_rule.h"
int main(int, char** v) {
    trt::PairRun r{};
    const long long nx = atoll(v[1]), ny = atoll(v[2]), n = atoll(v[3]);
    r.current = v[4][0] == 'c'; r.off = v[4][0] == 'o';
    const int w = r.current ? 56 : 60;
    r.nodes = n * nx * ny;
    r.columns = n * ((nx + w - 1) / w * w) * ny;
    r.tiled = n * ((nx + 31) / 32 * 32) * ny;
    r.elem = atoi(v[5]); r.general = atoi(v[6]); r.ghosts = atoi(v[7]);
    r.depth = atoi(v[8]); r.replayed = atoi(v[9]);
    r.mask = atoi(v[10]); r.crowded = atoi(v[11]); r.batch = atoi(v[12]);
    r.members = (int)n;
    r.padded = n * ((nx + 63) / 64 * 64) * ny;
    printf("%d", trt::two_steps_pay(r) ? 1 : 0);
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(SRC)
    exe = str(d / "rule")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2312_10318_gb300", "csrc"),
                    str(d / "rule.cpp"), "-o", exe], check=True)

    def call(nx, ny, n=1, mode="lagged", elem=4, general=0, ghosts=0, depth=1, replayed=1, mask=0, crowded=0,
             batch=0):
        return subprocess.run([exe, *(str(x) for x in (nx, ny, n, mode, elem, general, ghosts, depth, replayed, mask,
                                                       crowded, batch))],
                              check=True, capture_output=True, text=True).stdout == "1"
    return call


def test_periodic(rule):
    assert rule(64, 64) and rule(4096, 4096, 3) and rule(66, 64) and rule(66, 64, replayed=0)


def test_walls(rule):
    for elem in (2, 4):
        assert not rule(64, 64, 40, general=1, elem=elem) and not rule(512, 512, general=1, elem=elem)
        assert rule(1024, 1024, general=1, elem=elem) and rule(2048, 1024, general=1, elem=elem)
        assert not rule(64, 1024, 16, general=1, elem=elem) and rule(100, 1024, 16, general=1, elem=elem)
        assert rule(64, 64, general=1, ghosts=1, elem=elem)
    assert rule(512, 512, general=1, mode="off") and not rule(256, 256, general=1, mode="off")
    assert rule(32, 4096, 24, general=1, elem=4) and not rule(32, 4096, 24, general=1, elem=2)
    assert rule(32, 4096, 90, general=1, elem=2)


def test_several_lattices_launched_by_the_host(rule):
    for kw in (dict(general=1), dict(general=1, mask=1), dict(general=1, mode="off")):
        assert rule(130, 126, 8, replayed=0, **kw) and not rule(66, 64, 16, replayed=0, **kw)
        assert not rule(130, 126, 4, replayed=0, **kw)


def test_one_walled_lattice_launched_by_the_host(rule):
    assert rule(248, 1518, elem=2, general=1, replayed=0, batch=1)
    assert not rule(248, 1518, elem=2, general=1, replayed=0) and not rule(382, 380, general=1, replayed=0, batch=1)


def test_masks(rule):
    kw = dict(general=1, mask=1)
    assert not rule(1280, 1280, **kw) and rule(1536, 1536, **kw) and rule(100, 1024, 16, **kw)
    assert rule(768, 768, mode="off", **kw) and not rule(128, 128, 40, mode="off", **kw)
    assert rule(768, 768, crowded=1, **kw) and not rule(128, 128, 40, crowded=1, **kw)
    assert rule(64, 64, ghosts=1, **kw)


def test_current_phi(rule):
    for elem in (2, 4):
        assert rule(64, 64, mode="current", elem=elem, replayed=0)
        assert not rule(64, 64, mode="current", elem=elem) and not rule(512, 512, mode="current", elem=elem)
        assert rule(64, 64, 40, mode="current", elem=elem, depth=3)
        assert rule(768, 768, mode="current", elem=elem)
    assert rule(640, 640, mode="current", elem=4) and not rule(640, 640, mode="current", elem=2)
