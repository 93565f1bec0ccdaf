"""The double-float single-pair path against the oracle on two-body systems placed in each of its
regimes (needs a GB300): cleared runs and single sub-steps of the order-2 drift, the series to
order 6, sub-steps taken as several equal drifts, the FP64 Kepler solver, level changes of an
eccentric mutual orbit, fly-bys, subdivision by powers of two and not, a massless partner, a
heliocentric orbit far from circular, SI units.

Bars: positions to 1e-12 relative or within 100x the spread of the oracle's rounding-level
sensitivity twin, as for the single-pair path elsewhere; the oracle's sub-step count to 1 in 1,000
(equal below 1,000) and its depth to one level: a pair within rounding of a shell may be decided
differently from the oracle, which moves the few sub-steps below that shell.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402

G = 4.0 * math.pi ** 2
AU, MSUN = 1.495978707e11, 1.98841e30
YR = 2.0 * math.pi * math.sqrt(AU ** 3 / (6.6743e-11 * MSUN))

# a, e, inclination of the pair about the sun; separation, e of its own orbit; dt, M
CASES = {
    "order2_runs": (10.0, 0.0, 1e-5, 1e-3, 0.02, 0.05, {}),
    "order2_levels": (3.2, 0.0, 0.0, 2e-4, 0.6, 0.02, {}),
    "order6_runs": (5.0, 0.1, 0.02, 4e-3, 0.3, 0.5, {}),
    "two_drifts": (14.0, 0.0, 0.02, 4e-2, 0.1, 0.5, {}),
    "four_drifts": (6.0, 0.05, 0.02, 3e-2, 0.1, 0.5, {}),
    "sixteen_drifts": (5.5, 0.0, 0.5, 6e-2, 0.1, 0.5, {}),
    "kepler": (2.0, 0.2, 0.5, 5e-2, 0.1, 0.5, {}),
    "eccentric_heliocentric": (6.0, 0.6, 0.7, 1e-3, 0.4, 0.1, {}),
    "M3": (8.0, 0.01, 0.02, 1e-3, 0.4, 0.1, dict(M=3)),
    "M5_wide_shells": (8.0, 0.01, 0.02, 1e-3, 0.4, 0.1, dict(M=5, shell_ratio=2.9)),
    "M2_narrow_shells": (8.0, 0.01, 0.02, 1e-3, 0.4, 0.1, dict(M=2, shell_ratio=1.6)),
}


@pytest.fixture(scope="module")
def sy():
    import paper_2304_07325_gb300 as m
    from paper_2304_07325_gb300 import build
    build.build()
    return m


def _pair(a, e, inc, sep, eb, m, fly=1.0):
    xc, vc = disk.elements_to_state(a, e, inc, 0.7, 0.4, 2.0, G * (1.0 + m.sum()))
    xr, vr = disk.elements_to_state(sep, eb, 0.3, 0.5, 0.2, 1.1, G * m.sum())
    f = m[1] / m.sum()
    return (np.array([xc - f * xr, xc + (1.0 - f) * xr]),
            np.array([vc - f * fly * vr, vc + (1.0 - f) * fly * vr]))


def _check(orc, sy, x, v, m, radius, kw, steps=2):
    ref = orc.OracleSim(x, v, m, radius, params=orc.make_params(**kw))
    gpu = sy.System(x, v, m, radius, params=sy.default_params(**kw))
    pair = 0
    for _ in range(steps):
        twin = orc.OracleSim(x, v, m, radius, rhill=ref.rhill, params=orc.make_params(noise=1, **kw))
        twin.set_state(ref.x, ref.v)
        gpu.set_state(ref.x, ref.v)
        assert ref.step(1) >= 0 and twin.step(1) >= 0
        gpu.step(1)
        assert gpu.sync() >= 0
        st = gpu.stats()
        calls = sum(ref.level_calls[1:])
        assert abs(st.substeps - calls) <= calls // 1000 and abs(st.max_depth - ref.max_depth_seen) <= 1
        xg = gpu.get_state()[0]
        norm = np.linalg.norm(ref.x, axis=1)
        rel = np.linalg.norm(xg - ref.x, axis=1) / norm
        spread = np.linalg.norm(twin.x - ref.x, axis=1) / norm
        assert np.all(rel <= np.maximum(1e-12, 100.0 * spread)), (rel, spread)
        pair += st.pair_substeps
    assert pair > 0
    gpu.close()


@pytest.mark.parametrize("name", CASES)
def test_pair_in_each_regime(orc, sy, name):
    a, e, inc, sep, eb, dt, kw = CASES[name]
    m = np.array([3e-8, 2e-8])
    x, v = _pair(a, e, inc, sep, eb, m)
    _check(orc, sy, x, v, m, np.full(2, 1e-9), dict(dt=dt, **kw))


@pytest.mark.parametrize("what", ["fly_by", "massless_partner", "SI_units", "backwards"])
def test_pair_variants(orc, sy, what):
    m = np.array([3e-8, 2e-8])
    x, v = _pair(7.0, 0.02, 0.02, 1e-3, 0.3, m, fly=3.0 if what == "fly_by" else 1.0)
    kw = dict(dt=-0.05 if what == "backwards" else 0.05)
    if what == "massless_partner":
        m = np.array([3e-8, 0.0])
    if what == "SI_units":
        x, v, m, kw = x * AU, v * AU / YR, m * MSUN, dict(dt=0.05 * YR, G=6.6743e-11, m0=MSUN)
    _check(orc, sy, x, v, m, np.full(2, 1e-9 * (AU if what == "SI_units" else 1.0)), kw)


@pytest.mark.parametrize("a,e,dt", [(7.4, 0.0, 0.11), (5.0, 0.0, 0.133), (5.0, 0.0, 0.135), (6.0, 0.6, 0.05), (9.0, 0.3, 0.5)])
def test_series_to_order_10(orc, sy, a, e, dt):
    """Levels on both sides of s = 2e-6 (order 6 to 10) and of s = 1.28e-4 (order 10 to the Kepler
    solver), near pericentre of eccentric orbits too: a wide pair that stays on shallow levels."""
    m = np.array([3e-8, 2e-8])
    x, v = _pair(a, e, 0.02, 6e-3 * a, 0.1, m)
    _check(orc, sy, x, v, m, np.full(2, 1e-9), dict(dt=dt))
