"""State reads through each of their ways (needs a GB300): packed (small), straight into the caller's arrays
(large), staged in an allocation of the call (a pool with few pair slots), device arrays, and reads and
steps of one pool from two threads."""
import ctypes
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402


@pytest.mark.parametrize("n,pairs", [(1, 0), (100, 0), (3900, 0), (12000, 0), (500, 8), (12000, 8)])
def test_host_and_device_reads_agree(n, pairs):
    import torch

    import paper_2304_07325_gb300 as sy
    from paper_2304_07325_gb300 import build

    build.build()
    d = disk.planetesimal_disk(n, 60 + n)
    s = sy.System(d.x, d.v, d.m, d.radius, params=sy.default_params(dt=0.01, hill_scale=0.0, pair_capacity=pairs))
    s.step(1)
    host = s.get_state()
    dev = [torch.zeros(k, dtype=t, device="cuda") for k, t in ((3 * n, torch.float64), (3 * n, torch.float64),
                                                               (n, torch.float64), (n, torch.float64), (n, torch.int32))]
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    assert sy.lib().symba_get_state(s._h, *(ptr(t) for t in dev)) == sy.SYMBA_OK
    for a, b in zip(host, dev):
        assert np.array_equal(a.ravel(), b.cpu().numpy())
    assert np.array_equal(host[2], d.m) and np.array_equal(host[3], d.radius)
    s.close()


def test_reads_beside_steps_of_another_thread():
    import paper_2304_07325_gb300 as sy
    from paper_2304_07325_gb300 import build

    build.build()
    ds = [disk.planetesimal_disk(400, 80 + k) for k in range(2)]
    tiles = sum(((d.n + 31) // 32) ** 2 for d in ds)
    pool = sy.Pool(2, sum(d.n for d in ds), tiles)
    params = sy.default_params(dt=0.01, hill_scale=0.0)          # no encounters, so no mergers
    slots = [pool.admit(d.x, d.v, d.m, d.radius, params=params) for d in ds]
    bad = []

    def read():
        for _ in range(100):
            for slot, d in zip(slots, ds):
                x, v, m, r, a = pool.get_state(slot)
                if not (np.isfinite(x).all() and np.array_equal(r, d.radius) and np.array_equal(m, d.m)):
                    bad.append(slot)
    t = threading.Thread(target=read)
    t.start()
    for _ in range(20):
        pool.step(1)
    t.join()
    assert pool.sync() >= 0 and not bad
    pool.close()
