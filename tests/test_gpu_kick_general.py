"""Where the double-float pair kick of FP64 systems hands a macro-tile, or a chunk of the field rectangle, to
its FP64 form (needs a GB300): systems with a body far from the rest, at set-up or through set_state, pairs
closer than FP32's range allows, and the same at the edges of tiles and with flagged pairs.

Reference: one step without encounters in extended precision (numpy's long double) from the state the
library holds.  With e = 2^-53 the bar on a body's velocity is 16 e (|v| + K + X) + 2^-44 K.  16 e covers the
roundings of v and the eight of a pair's force in FP64; 2^-44 K is the double-float form's own bar, K the
sum of the magnitudes of both kicks' pair terms and X the same sum weighted by (|x_i| + |x_j|) / r, the
effect of the roundings of x."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402

G = 4.0 * math.pi ** 2
LD = np.longdouble


@pytest.fixture(scope="module")
def sy():
    import paper_2304_07325_gb300 as m
    from paper_2304_07325_gb300 import build
    build.build()
    return m


def _kepler_ld(mu, dt, x, v):
    """Two-body motion by universal variables (n dt of a few radians at most)."""
    r0 = np.sqrt((x * x).sum(1))
    u = (x * v).sum(1)
    al = 2 * mu / r0 - (v * v).sum(1)
    s = np.full(len(x), LD(dt)) / r0
    for _ in range(60):
        z = al * s * s
        c = [np.zeros_like(z) for _ in range(4)]
        for k in range(4):
            t = np.ones_like(z) / LD(math.factorial(k))
            for j in range(40):
                c[k] = c[k] + t
                t = -t * z / LD((2 * j + k + 1) * (2 * j + k + 2))
        G1, G2, G3 = s * c[1], s * s * c[2], s * s * s * c[3]
        r = r0 * c[0] + u * G1 + mu * G2
        s = s - (r0 * G1 + u * G2 + mu * G3 - dt) / r
    f1, g, fd, gd1 = -mu * G2 / r0, dt - mu * G3, -mu * G1 / (r * r0), -mu * G2 / r
    return x + f1[:, None] * x + g[:, None] * v, v + fd[:, None] * x + gd1[:, None] * v


def step_ld(x, v, m, nm, dt):
    """One step without encounters; also K and X of both kicks per body (over |v|'s unit)."""
    x, v, m, h = x.astype(LD), v.astype(LD), m.astype(LD), LD(dt) / 2
    K, X = np.zeros(len(m), dtype=LD), np.zeros(len(m), dtype=LD)

    def kick(v):
        a = np.zeros_like(x)
        size = np.sqrt((x * x).sum(1))
        for i in range(nm):
            d = x[i] - x
            r2 = (d * d).sum(1)
            r2[i] = np.inf
            s = LD(G) * m[i] / (r2 * np.sqrt(r2))
            a += s[:, None] * d
            K[:] += h * s * np.sqrt(np.where(np.isfinite(r2), r2, 0))
            X[:] += h * s * (size + size[i])
        return v + h * a
    sun = lambda: h * (m[:, None] * v).sum(0)
    x = x + sun()
    v = kick(v)
    x, v = _kepler_ld(LD(G), LD(dt), x, v)
    v = kick(v)
    return x + sun(), v, K, X


def bar(v, K, X, df=2.0 ** -44, c=16):
    return c * 2.0 ** -53 * (np.sqrt((v * v).sum(1)) + K + X) + df * K


def check(sy, x, v, m, nm, dt, state=None, df=2.0 ** -44, c=16):
    gpu = sy.System(x, v, m, np.zeros(len(m)), n_massive=nm, params=sy.default_params(hill_scale=0.0, dt=dt))
    if state is not None:
        gpu.set_state(*state)
    x0, v0 = gpu.get_state()[:2]
    xr, vr, K, X = step_ld(x0, v0, m, nm, dt)
    gpu.step(1)
    assert gpu.sync() >= 0
    xg, vg = gpu.get_state()[:2]
    gpu.close()
    err = np.sqrt(((vg - vr) ** 2).sum(1))
    b = bar(vr, K, X, df, c)
    assert np.all(err <= b), (int(np.argmax(err / b)), float((err / b).max()))
    assert np.all(np.sqrt(((xg - xr) ** 2).sum(1)) <= 2e-14 * np.sqrt((xr * xr).sum(1)) + dt * b)


def heavy_disk(n, seed, nf=0, mass=1e-3):
    d = disk.planetesimal_disk(n, seed, n_field=nf)
    m = np.where(d.m > 0.0, mass * (0.5 + 0.5 * d.m / d.m.max()), 0.0)
    return d.x.copy(), d.v.copy(), m


@pytest.mark.parametrize("who", ["massive", "field"])
@pytest.mark.parametrize("factor", [1e7, 1e9, 1e11, 1e13])
def test_a_body_far_from_the_rest(sy, who, factor):
    x, v, m = heavy_disk(150, 31, 80)
    k = 70 if who == "massive" else 200
    x[k] *= factor
    v[k] /= math.sqrt(factor)
    check(sy, x, v, m, 150, 0.1)


@pytest.mark.parametrize("factor", [1e7, 1e12])
def test_a_body_that_goes_far_after_set_up(sy, factor):
    x, v, m = heavy_disk(150, 31, 80)
    s = sy.System(x, v, m, np.zeros(len(m)), n_massive=150)
    xs, vs = s.get_state()[:2]
    s.close()
    for k in (70, 200):
        xs[k] *= factor
        vs[k] /= math.sqrt(factor)
    check(sy, x, v, m, 150, 0.1, state=(xs, vs))


def test_a_state_of_another_scale(sy):
    x, v, m = heavy_disk(150, 31, 80)
    check(sy, x, v, m, 150, 0.1, state=(x * 2.0 ** 70, v * 2.0 ** -35))


@pytest.mark.parametrize("n,nf", [(1, 0), (2, 0), (31, 0), (33, 0), (64, 0), (65, 0), (127, 0), (129, 0), (193, 0), (257, 0),
                                  (1, 40), (33, 31), (40, 100), (128, 65), (129, 33), (161, 300)])
def test_tile_edges_in_fp64(sy, n, nf):
    """Every macro-tile and chunk has a member at 1e9 times its distance."""
    x, v, m = heavy_disk(n, 900 + n, nf)
    for k in range(0, n + nf, 32):
        x[k] *= 1e9
        v[k] /= math.sqrt(1e9)
    check(sy, x, v, m, n, 0.1)


def test_pairs_closer_than_the_fp32_range(sy):
    """Pairs of negligible mass 3e-13 apart: a step without them, to what the roundings of x make of it."""
    x, v, m = heavy_disk(100, 7, 60, mass=1e-30)
    for i, j in ((3, 90), (40, 41), (10, 130)):
        x[j] = x[i] + 3e-13
        v[j] = v[i]
    gpu = sy.System(x, v, m, np.zeros(len(m)), n_massive=100, params=sy.default_params(hill_scale=0.0, dt=0.1))
    x0, v0 = gpu.get_state()[:2]
    xr, vr, K, X = step_ld(x0, v0, m, 100, 0.1)
    gpu.step(1)
    assert gpu.sync() >= 0
    xg, vg = gpu.get_state()[:2]
    gpu.close()
    # (a separation of 3e-13 at 20 AU moves by up to a few per cent with the roundings of x)
    assert np.all(np.sqrt(((vg - vr) ** 2).sum(1)) <= 1e-14 * np.sqrt((vr * vr).sum(1)) + 0.5 * K)


@pytest.mark.parametrize("nf", [0, 200])
def test_flagged_pairs_beside_a_far_body(orc, sy, nf):
    """Encounters in macro-tiles and chunks that are taken in FP64: listed once, weighted in both kicks."""
    d = disk.planetesimal_disk(300, 77, n_field=nf)
    x, v = d.x.copy(), d.v.copy()
    m = d.m * 30.0
    for k in range(5, 300 + nf, 32):
        x[k] *= 1e11
        v[k] /= math.sqrt(1e11)
    radius = np.full(len(m), 1e-7)
    ref = orc.OracleSim(x, v, m, radius, n_massive=300, params=orc.make_params(dt=0.05))
    twin = orc.OracleSim(x, v, m, radius, n_massive=300, rhill=ref.rhill, params=orc.make_params(noise=1, dt=0.05))
    gpu = sy.System(x, v, m, radius, n_massive=300, params=sy.default_params(dt=0.05))
    assert ref.step(1) >= 0 and twin.step(1) >= 0
    gpu.step(1)
    assert gpu.sync() >= 0
    pairs = gpu.enc_groups()[0]
    want = ref.enc_groups()[0]
    assert len(pairs) >= 10 and np.array_equal(np.asarray(pairs), np.asarray(want))
    xg, vg, mg, _, ag = gpu.get_state()
    gpu.close()
    assert np.array_equal(ag, ref.alive) and np.array_equal(mg, ref.m)
    live = ref.alive != 0
    for a, b, t in ((xg, ref.x, twin.x), (vg, ref.v, twin.v)):
        rel = (np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1))[live]
        spread = (np.linalg.norm(t - b, axis=1) / np.linalg.norm(b, axis=1))[live]
        assert np.all(rel <= np.maximum(1e-13, 100.0 * spread)), float((rel / np.maximum(1e-13, 100.0 * spread)).max())


def test_neighbours_and_schedules_change_no_bit(sy):
    """Systems with macro-tiles taken in FP64, alone, in one pool with an ordinary one, and with several
    macro-tiles per grab."""
    ds = []
    for n, nf, far in ((300, 80, True), (500, 0, False), (700, 200, True)):
        x, v, m = heavy_disk(n, 50 + n, nf)
        if far:
            for k in range(20, n + nf, 150):
                x[k] *= 1e9
                v[k] /= math.sqrt(1e9)
        ds.append((x, v, m, n))
    params = sy.default_params(hill_scale=0.0, dt=0.05)
    alone = []
    for x, v, m, n in ds:
        s = sy.System(x, v, m, np.zeros(len(m)), n_massive=n, params=params)
        s.step(3)
        assert s.sync() >= 0
        alone.append(s.get_state())
        s.close()
    tiles = sum(((len(m) + 31) // 32) ** 2 for _, _, m, _ in ds)
    for per_item in (1, 16):
        pool = sy.Pool(3, sum(len(m) for _, _, m, _ in ds), tiles)
        slots = [pool.admit(x, v, m, np.zeros(len(m)), n_massive=n, params=params) for x, v, m, n in ds]
        pool.schedule = dict(pool.schedule, kick_tiles_per_item=per_item)
        pool.step(3)
        assert pool.sync() >= 0
        for k, want in zip(slots, alone):
            assert all(np.array_equal(a, b) for a, b in zip(pool.get_state(k), want))
        pool.close()
