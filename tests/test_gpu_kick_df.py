"""The double-float pair kick of FP64 systems at the edges of its tiles, macro-tiles and field chunks,
in other units, with a far and with a heavy body (needs a GB300): one step without encounters
(hill_scale = 0) against the oracle.

Bar on every body's velocity: 2e-14 of |v| (the Kepler and sun drifts, as elsewhere) plus 2^-44 of the
sum of its pair kicks' magnitudes (2^-46 per product and sum of the pair arithmetic)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402

G = 4.0 * math.pi ** 2
AU, MSUN = 1.495978707e11, 1.98841e30
YR = 2.0 * math.pi * math.sqrt(AU ** 3 / (6.6743e-11 * MSUN))


@pytest.fixture(scope="module")
def sy():
    import paper_2304_07325_gb300 as m
    from paper_2304_07325_gb300 import build
    build.build()
    return m


def _check(orc, sy, x, v, m, nm, G, kw):
    n = len(m)
    radius = np.zeros(n)
    ref = orc.OracleSim(x, v, m, radius, n_massive=nm, params=orc.make_params(hill_scale=0.0, **kw))
    gpu = sy.System(x, v, m, radius, n_massive=nm, params=sy.default_params(hill_scale=0.0, **kw))
    kick = np.zeros(n)
    for i in range(nm):
        r2 = ((x - x[i]) ** 2).sum(1)
        r2[i] = np.inf
        kick += G * m[i] / r2
    assert ref.step(1) >= 0
    gpu.step(1)
    assert gpu.sync() >= 0
    st = gpu.stats()
    assert st.n_pairs == 0
    xg, vg = gpu.get_state()[:2]
    err = np.linalg.norm(vg - ref.v, axis=1)
    bar = 2e-14 * np.linalg.norm(ref.v, axis=1) + 2.0 ** -44 * abs(kw["dt"]) * kick
    assert np.all(err <= bar), (int(np.argmax(err / bar)), float((err / bar).max()))
    assert np.abs(xg - ref.x).max() <= 2e-14 * np.abs(ref.x).max()
    gpu.close()


@pytest.mark.parametrize("n,nf", [(1, 0), (2, 0), (31, 0), (33, 0), (64, 0), (65, 0), (127, 0), (129, 0), (193, 0),
                                  (257, 0), (1, 40), (33, 31), (40, 100), (128, 65), (129, 33), (161, 300)])
def test_edges(orc, sy, n, nf):
    d = disk.planetesimal_disk(n, 900 + n, n_field=nf)
    _check(orc, sy, d.x, d.v, d.m, n, G, dict(dt=0.1))


@pytest.mark.parametrize("what", ["SI", "far_body", "heavy_body", "tilted"])
def test_units_and_spread(orc, sy, what):
    d = disk.planetesimal_disk(150, 31, n_field=50)
    x, v, m, g, kw = d.x.copy(), d.v.copy(), d.m.copy(), G, dict(dt=0.1)
    if what == "SI":
        x, v, m, g, kw = x * AU, v * AU / YR, m * MSUN, 6.6743e-11, dict(dt=0.1 * YR, G=6.6743e-11, m0=MSUN)
    if what == "far_body":
        x[70] *= 3e4
        v[70] /= math.sqrt(3e4)
    if what == "heavy_body":
        m[3] = 1e-3
    if what == "tilted":
        q = np.linalg.qr(np.random.RandomState(4).randn(3, 3))[0]
        x, v = x @ q.T, v @ q.T
    _check(orc, sy, x, v, m, d.n_massive, g, kw)
