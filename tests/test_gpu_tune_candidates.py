"""The autotuner times each kick schedule once: the CTAs per SM that are resident together (which is what a pool
starts with) times the five grab sizes; a schedule with more of them is accepted, and is the same kick
(needs a GB300)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_kick_candidates(precision):
    import paper_2304_07325_gb300 as sy
    from paper_2304_07325_gb300 import build

    build.build()
    d = disk.planetesimal_disk(600, 4300)
    states = []
    for kb in (0, 4):
        pool = sy.Pool(1, d.n, ((d.n + 31) // 32) ** 2, precision=precision)
        slot = pool.admit(d.x, d.v, d.m, d.radius)
        resident = pool.schedule["kick_blocks_per_sm"]
        if kb:
            pool.schedule = dict(pool.schedule, kick_blocks_per_sm=kb)
        assert pool.autotune(reps=1)["kick_candidates"] == 5 * resident
        pool.step(1)
        assert pool.sync() >= 0
        states.append(pool.get_state(slot))
        pool.close()
    assert all(np.array_equal(a, b) for a, b in zip(*states))
