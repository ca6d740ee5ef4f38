"""The bench's launch counts of runs that take two steps per launch (host only)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("steps", [1, 2, 3, 31, 32, 33, 64, 100])
@pytest.mark.parametrize("odd", [False, True])
@pytest.mark.parametrize("batch", [False, True])
def test_runs_of_two_step_launches(steps, odd, batch):
    """Against the sequence the library launches: Phi lagged, a single step to an odd
    level, then twos; a batch replays runs of 32 steps after that single step, or,
    where the run is just 32, one whose twos are even in number.  Phi at the current
    level: twos from any level."""
    sys.path.insert(0, ROOT)
    import bench

    def library(n, odd, graph):
        pairs, level = 0, odd
        if batch and not level and n > 32:
            n, level = n - 1, True
        if batch:
            while n >= 32:
                pairs += 16 if level else 14
                n -= 32
        if n and not level:
            n, level = n - 1, True
        return pairs + n // 2

    pairs, singles = bench.two_step_run(steps, odd, "lagged", batch)
    assert pairs == library(steps, odd, batch) and 2 * pairs + singles == steps
    assert bench.two_step_run(steps, odd, "off", batch) == (pairs, singles)
    assert bench.two_step_run(steps, odd, "current", batch) == (steps // 2, steps % 2)


def test_launches_of_a_run():
    """Three lattices: with Phi at the current level a batch takes one launch for two
    steps of all of them, and as many as its single-step kernel takes for an odd one."""
    sys.path.insert(0, ROOT)
    import bench
    assert bench.run_launches("batch", ["ab_tma"] * 3, True, 100, True, "current") == 50
    assert bench.run_launches("batch", ["ab_tma"] * 3, True, 101, False, "current") == 50 + 3
    assert bench.run_launches("single", ["ab_column"] * 3, True, 100, False, "current") == 150
    assert bench.run_launches("batch", ["ab_tma"] * 3, False, 100, False, "current") == 300
    assert bench.run_launches("batch", ["aa_vector"] * 3, True, 100, True, "lagged") == 50
    assert bench.run_launches("batch", ["aa"] * 100, True, 10, True, "lagged") == 10
    assert "k_step_ab_pair" in bench.TWO_STEP_NAMES["current"] and "k_step_pair" in bench.TWO_STEP_NAMES["lagged"]
