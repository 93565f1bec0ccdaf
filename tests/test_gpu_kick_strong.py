"""Kicks that are a large part of the velocity (needs a GB300), from forces far below the line at which a
macro-tile or a field chunk is taken in FP64 to far above it: heavy bodies at 0.05 to some AU, and bodies
of several m0, whose kick in a hundredth of a year is several |v|.

Reference: one step without encounters in extended precision.  Bar on every body's velocity, without the
double-float form's own term: 16 e (|v| + K + X) as in test_gpu_kick_general, e = 2^-53, and 8 e (|v| + K + X)
where the step is so short that the Kepler drift's roundings do not count: 4 e |v| of its and the kicks'
roundings, 5 e K of a force's eight roundings in FP64, 6 e X of positions rounded once before the first
kick and five times before the second.  A kick good to 2^-46 of K fails the latter, where K is several |v|."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_kick_general import G, bar, check, heavy_disk, step_ld  # noqa: E402

from paper_2304_07325_gb300 import disk  # noqa: E402


@pytest.fixture(scope="module")
def sy():
    import paper_2304_07325_gb300 as m
    from paper_2304_07325_gb300 import build
    build.build()
    return m


def few(n, nf, mass, seed, apart=0.15):
    """n heavy bodies and nf field particles around 1 AU, the heavy ones some `apart` from one another."""
    rng = np.random.RandomState(seed)
    x, v = [], []
    for k in range(n + nf):
        a, b = disk.elements_to_state(1.0 + 0.3 * rng.rand(), 0.1 * rng.rand(), 0.1 * rng.rand(), 6.28 * rng.rand(),
                                      6.28 * rng.rand(), apart * ((k if apart < 1.0 else min(k, n)) + 0.3 * rng.rand()), G)
        x.append(a)
        v.append(b)
    m = np.zeros(n + nf)
    m[:n] = mass * (0.3 + 0.7 * rng.rand(n))
    return np.array(x), np.array(v), m


@pytest.mark.parametrize("n,nf", [(2, 0), (3, 0), (5, 40)])
@pytest.mark.parametrize("mass", [1e-6, 1e-4, 1e-3, 1e-2, 5e-2])
def test_a_few_heavy_bodies(sy, n, nf, mass):
    for seed in range(8):
        x, v, m = few(n, nf, mass, seed)
        check(sy, x, v, m, n, 0.1, df=0.0)


@pytest.mark.parametrize("n,nf", [(2, 0), (3, 0)])
@pytest.mark.parametrize("mass", [1.0, 3.0, 10.0])
def test_kicks_above_the_velocity(sy, n, nf, mass):
    for seed in range(16):
        x, v, m = few(n, nf, mass, seed, apart=1.5)
        check(sy, x, v, m, n, 0.01, df=0.0, c=8)


@pytest.mark.parametrize("mass", [1e-5, 1e-3, 1e-2])
@pytest.mark.parametrize("n,nf", [(33, 0), (150, 80), (300, 500)])
def test_heavy_disks(sy, n, nf, mass):
    x, v, m = heavy_disk(n, 40 + n, nf, mass)
    check(sy, x, v, m, n, 0.5, df=0.0)


def test_the_bar_sees_a_46_bit_kick():
    """The bar itself, on the CPU's own numbers: forces good to 46 bits miss it, FP64 forces do not."""
    worst = {46: 0.0, 53: 0.0}
    for seed in range(16):
        x, v, m = few(2, 0, 10.0, seed, apart=1.5)
        xr, vr, K, X = step_ld(x, v, m, 2, 0.01)
        for bits in worst:
            worst[bits] = max(worst[bits], float((K * 2.0 ** -bits / bar(vr, K, X, 0.0, 8)).max()))
    assert worst[46] > 2.0 and worst[53] < 0.2
