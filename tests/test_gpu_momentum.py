"""Total momentum and closing sun drift (needs a GB300): the single-kernel form for systems of up to 2,048
bodies and the three-kernel form for larger ones round the same exact sum, so a small system steps to
the same bits alone and in a pool whose largest system takes the other form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402


@pytest.mark.parametrize("sizes", [(1, 2049), (100, 3000), (2048, 2049), (31, 33)])
@pytest.mark.parametrize("precision", [0, 1])
def test_small_system_alone_and_beside_a_large_one(sizes, precision):
    import paper_2304_07325_gb300 as sy
    from paper_2304_07325_gb300 import build

    build.build()
    ds = [disk.planetesimal_disk(n, 700 + n, n_field=7 * k) for k, n in enumerate(sizes)]
    params = sy.default_params(dt=0.1, precision=precision)
    tiles = sum(((d.n + 31) // 32) * ((d.n_massive + 31) // 32) for d in ds)
    pool = sy.Pool(len(ds), sum(d.n for d in ds), tiles, precision)
    slots = [pool.admit(d.x, d.v, d.m, d.radius, params=params, n_massive=d.n_massive) for d in ds]
    alone = [sy.System(d.x, d.v, d.m, d.radius, n_massive=d.n_massive, params=params) for d in ds]
    pool.step(3)
    assert pool.sync() >= 0
    for slot, s in zip(slots, alone):
        s.step(3)
        assert s.sync() >= 0
        for a, b in zip(pool.get_state(slot), s.get_state()):
            assert np.array_equal(a, b)
        s.close()
    pool.close()
