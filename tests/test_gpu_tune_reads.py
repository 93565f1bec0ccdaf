"""State reads of one thread beside the autotuner in another (needs a GB300): the tuner's trial steps use the
scratch in which reads stage and change the state until it is put back, so a read returns the state as it
was before the call, never a trial state or a trial step's forces."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_reads_beside_the_autotuner(precision):
    import paper_2304_07325_gb300 as sy
    from paper_2304_07325_gb300 import build

    build.build()
    ds = [disk.planetesimal_disk(n, 4200 + n) for n in (500, 900)]
    tiles = sum(((d.n + 31) // 32) ** 2 for d in ds)
    pool = sy.Pool(2, sum(d.n for d in ds), tiles, precision=precision)
    slots = [pool.admit(d.x, d.v, d.m, d.radius) for d in ds]
    pool.step(1)
    assert pool.sync() >= 0
    want = [pool.get_state(s) for s in slots]
    stop, bad, reads = threading.Event(), [], [0]

    def read():
        while not stop.is_set():
            for s, w in zip(slots, want):
                if not all(np.array_equal(a, b) for a, b in zip(pool.get_state(s), w)):
                    bad.append(s)
                reads[0] += 1
    t = threading.Thread(target=read)
    t.start()
    tuned = [pool.autotune(reps=1) for _ in range(5)]
    stop.set()
    t.join()
    assert all(r["identical"] == 1 for r in tuned) and reads[0] > 0 and not bad
    assert all(np.array_equal(a, b) for s, w in zip(slots, want) for a, b in zip(pool.get_state(s), w))
    pool.close()
