"""symba_profile_step times the closing sun drift as a phase of its own, after the total momentum, for systems
on either side of the size from which on a step takes the two in one kernel, and leaves the bits that
symba_step leaves (needs a GB300)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

G = 4.0 * math.pi ** 2


@pytest.fixture(scope="module")
def sy():
    import paper_2304_07325_gb300 as m
    from paper_2304_07325_gb300 import build
    build.build()
    return m


def circular(n, seed):
    rng = np.random.RandomState(seed)
    a, t = 5.0 + 15.0 * rng.rand(n), 2.0 * math.pi * rng.rand(n)
    w = np.sqrt(G / a)
    return (np.stack([a * np.cos(t), a * np.sin(t), 0.0 * a], 1), np.stack([-w * np.sin(t), w * np.cos(t), 0.0 * a], 1))


def test_the_closing_drift_has_its_own_phase(sy):
    n = 1000000
    x, v = circular(n, 1)
    m = np.zeros(n)
    m[:10] = 1e-6
    s = sy.System(x, v, m, np.zeros(n), n_massive=10, params=sy.default_params(dt=0.01, hill_scale=0.0, pair_capacity=64))
    ph = np.min([s.profile_step(1) for _ in range(6)], axis=0)
    s.close()
    # the opening drift reads and writes about 160 bytes a body, the closing one 52: without any kernel
    # between its events phase 9 would be 2 us beside some 40
    assert ph[9] > 0.15 * ph[0], ph


@pytest.mark.parametrize("n", [1, 31, 500, 2048, 2049, 3000])
def test_the_same_bits_as_a_step(sy, n):
    x, v = circular(n, n)
    m = np.full(n, 1e-9)
    a, b = (sy.System(x, v, m, np.zeros(n), params=sy.default_params(dt=0.1, hill_scale=0.0)) for _ in range(2))
    a.step(3)
    b.profile_step(3)
    assert a.sync() >= 0 and b.sync() >= 0
    assert all(np.array_equal(p, q) for p, q in zip(a.get_state(), b.get_state()))
    a.close()
    b.close()
