"""The Kepler drift over its branches (needs a GB300): Taylor series to 1/2, doubled series to 1, library
sine beyond, several orbits, near-parabolic and hyperbolic orbits, zero and backward-looking phases, and
units outside the FP32 seeds' range, against the same f and g functions in extended precision.

Bar on every body: the change that relative perturbations of 2^-53 in each of x, v, mu and dt bring,
added up and times 8 (about 10 roundings lead to each of the solver's elements), plus 2^-50 of |x|, |v|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402

LD = np.longdouble


def _drift(mu, dt, x, v):
    """Exact drift of (n, 3) states in extended precision, by bisected Newton in a universal variable."""
    r0, v2, u = np.sqrt((x * x).sum(1)), (v * v).sum(1), (x * v).sum(1)
    al = 2 * mu / r0 - v2
    ell = al > 0
    k = np.sqrt(np.abs(al))

    def G(s):                            # G_0..G_3
        w = k * s
        sm = np.abs(w) < LD(1) / 8
        z = np.where(ell, 1, -1) * w * w
        c2, c3, t2, t3 = (np.zeros_like(w) for _ in range(4))
        t2 += LD(1) / 2
        t3 += LD(1) / 6
        for j in range(12):
            c2, c3 = c2 + t2, c3 + t3
            t2, t3 = t2 * -z / ((2 * j + 3) * (2 * j + 4)), t3 * -z / ((2 * j + 4) * (2 * j + 5))
        wm = np.where(sm, 1, w)
        we, wh = np.where(ell, wm, 1), np.where(ell, 1, np.minimum(wm, 50))
        c2b = np.where(ell, 2 * np.sin(we / 2) ** 2 / we ** 2, 2 * np.sinh(wh / 2) ** 2 / wh ** 2)
        c3b = np.where(ell, (we - np.sin(we)) / we ** 3, (np.sinh(wh) - wh) / wh ** 3)
        c2, c3 = np.where(sm, c2, c2b), np.where(sm, c3, c3b)
        zz = np.where(ell, 1, -1) * w * w
        return 1 - zz * c2, s * (1 - zz * c3), s * s * c2, s ** 3 * c3
    lo, hi = np.zeros_like(r0), dt / r0
    for _ in range(80):
        g = G(hi)
        hi = np.where(r0 * g[1] + u * g[2] + mu * g[3] < dt, 2 * hi, hi)
    s = (lo + hi) / 2
    for _ in range(160):
        g = G(s)
        F, Fp = r0 * g[1] + u * g[2] + mu * g[3] - dt, r0 * g[0] + u * g[1] + mu * g[2]
        lo, hi = np.where(F > 0, lo, s), np.where(F > 0, s, hi)
        n = s - F / Fp
        s = np.where((n > lo) & (n < hi), n, (lo + hi) / 2)
    g = G(s)
    r = r0 * g[0] + u * g[1] + mu * g[2]
    c = lambda a: a[:, None]
    return (x + c(-mu * g[2] / r0) * x + c(dt - mu * g[3]) * v, v + c(-mu * g[1] / (r * r0)) * x + c(-mu * g[2] / r) * v)


def _states(what, dt, G, unit):
    rng = np.random.default_rng(len(what))
    e = {"round": 0.0, "disk": 0.05, "eccentric": 0.7, "comet": 0.97}.get(what, 0.0)
    # n dt over 4e-4 .. 30, thick at the borders 1/2, 1 and 3 of the branches
    nh = np.concatenate([np.geomspace(4e-4, 30.0, 150), 0.5 + np.linspace(-1e-3, 1e-3, 20), 1.0 + np.linspace(-1e-3, 1e-3, 20),
                         3.0 + np.linspace(-0.2, 0.2, 20)])
    xs, vs = [], []
    for h in nh:
        a = (G * (dt / h) ** 2) ** (1.0 / 3.0)
        x, v = disk.elements_to_state(a, e * rng.uniform(0.5, 1.0), 0.2, *rng.uniform(0.0, 6.28, 3), G)
        x, v = np.asarray(x), np.asarray(v)
        if what == "unbound":
            v = v * np.sqrt(2.0) * rng.choice([1.0 + 1e-9, 1.05, 3.0])
        xs.append(x)
        vs.append(v)
    return np.array(xs), np.array(vs)


def _bars(mu, dt, x, v):
    X, V = _drift(LD(mu), LD(dt), x.astype(LD), v.astype(LD))
    nx, nv = (np.sqrt((a * a).sum(1)) for a in (X, V))
    bx, bv = nx * LD(2) ** -50, nv * LD(2) ** -50
    for c in range(8):
        p = [LD(mu), LD(dt), x.astype(LD), v.astype(LD)]
        f = 1 + LD(2) ** -53
        if c < 6:
            p[2 + c // 3] = p[2 + c // 3].copy()
            # a rounding of |x| (|v|), not of a small component of it
            p[2 + c // 3][:, c % 3] += np.sqrt((p[2 + c // 3] ** 2).sum(1)) * LD(2) ** -53
        else:
            p[c - 6] = p[c - 6] * f
        Xp, Vp = _drift(*p)
        bx, bv = bx + 8 * np.sqrt(((Xp - X) ** 2).sum(1)), bv + 8 * np.sqrt(((Vp - V) ** 2).sum(1))
    return X, V, bx, bv


@pytest.mark.parametrize("what,unit", [("round", 1.0), ("disk", 1.0), ("eccentric", 1.0), ("comet", 1.0), ("unbound", 1.0),
                                       ("disk", 1e25), ("disk", 1e-25)])
def test_against_extended_precision(what, unit):
    import paper_2304_07325_gb300 as sy
    from paper_2304_07325_gb300 import build

    build.build()
    G, dt = sy.default_params().G, 0.5
    x, v = _states(what, dt, G, unit)
    x, v, G = x * unit, v * unit, G * unit ** 3
    n = len(x)
    s = sy.System(x, v, np.full(n, 1e-40), np.zeros(n), n_massive=0,
                  params=sy.default_params(dt=dt, G=G, m0=1.0, hill_scale=0.0), rhill=np.zeros(n))
    x, v = s.get_state()[:2]
    X, V, bx, bv = _bars(G, dt, x, v)
    s.step(1)
    assert s.sync() >= 0
    xg, vg = s.get_state()[:2]
    s.close()
    ex, ev = np.sqrt(((xg - X) ** 2).sum(1)) / bx, np.sqrt(((vg - V) ** 2).sum(1)) / bv
    assert np.all(ex <= 1.0) and np.all(ev <= 1.0), (float(ex.max()), float(ev.max()), int(np.argmax(ex)))
