"""The recursion of groups of several pairs in one warp's lanes against the oracle (needs a GB300): two
close pairs at once, three bodies at once, groups that come down to 32 bodies and pairs only at deeper
levels (from shared and from global memory), mergers inside a group, other partition orders and
subdivisions, backwards, SI units, and units outside the double-float range (general FP64 path).

Bars: those of the single-pair tests, positions to 1e-12 relative or within 100x the spread of the
oracle's rounding-level sensitivity twin, depth to one level, mergers equal, and sub-steps to 1
in 1,000 (at most the oracle's where a level has several components, which it counts one by one)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402

G = 4.0 * math.pi ** 2
AU, MSUN = 1.495978707e11, 1.98841e30
YR = 2.0 * math.pi * math.sqrt(AU ** 3 / (6.6743e-11 * MSUN))


def _binary(a, phase, sep, eb, m, turn=0.4):
    xc, vc = disk.elements_to_state(a, 0.001, 1e-4, 0.7, 0.0, phase, G * (1.0 + m.sum()))
    xr, vr = disk.elements_to_state(sep, eb, 0.3, 0.5, 0.2, turn, G * m.sum())
    f = m[1] / m.sum()
    return [xc - f * xr, xc + (1.0 - f) * xr], [vc - f * vr, vc + (1.0 - f) * vr]


def system(kind):
    """x, v, m of a group: R_0 is about 0.25 between two bodies of 3e-8 at a = 8."""
    m2 = np.array([3e-8, 2e-8])
    x, v, m = [], [], []

    def put(xs, vs, ms):
        x.extend(xs)
        v.extend(vs)
        m.extend(ms)

    def single(a, phase, e=0.002):
        xs, vs = disk.elements_to_state(a, e, 1e-3, 0.7, 0.0, phase, G)
        put([xs], [vs], [2e-8])
    if kind in ("two_binaries", "binaries_and_field"):
        put(*_binary(8.0, 0.0, 2e-3, 0.3, m2), m2)
        put(*_binary(8.05, 0.01, 3e-3, 0.1, m2, 1.3), m2)
    if kind == "binaries_and_field":
        for k in range(5):
            single(7.95 + 0.02 * k, 0.005 * k)
    if kind == "triple":
        put(*_binary(8.0, 0.0, 4e-3, 0.2, m2), m2)
        xt, vt = _binary(8.0, 0.0, 2e-2, 0.1, np.array([5e-8, 2e-8]), 2.0)
        x[0], x[1] = (np.asarray(p) + (np.asarray(xt[0]) - 0.6 * np.asarray(x[0]) - 0.4 * np.asarray(x[1])) for p in (x[0], x[1]))
        vc = 0.6 * np.asarray(v[0]) + 0.4 * np.asarray(v[1])
        v[0], v[1] = (np.asarray(p) + (np.asarray(vt[0]) - vc) for p in (v[0], v[1]))
        put([xt[1]], [vt[1]], [2e-8])
    if kind == "shared_view":               # at most 32 bodies, 33 to 64 pairs
        put(*_binary(8.0, 0.0, 2e-3, 0.3, m2), m2)
        put(*_binary(8.04, 0.008, 5e-3, 0.3, m2), m2)
        for k in range(6):
            single(7.93 + 0.025 * k, 0.004 * (k + 1))
    if kind == "global_view":               # more than 32 bodies
        put(*_binary(8.0, 0.0, 2e-3, 0.3, m2), m2)
        put(*_binary(8.0, 0.2, 3e-3, 0.3, m2), m2)
        for k in range(38):
            single(8.0 + 0.03 * (-1) ** k, 0.0125 * (k + 1) - 0.1)
    return np.array(x, dtype=np.float64), np.array(v, dtype=np.float64), np.array(m)


CASES = {
    "two_binaries": ("two_binaries", 0.1, {}, 1e-9),
    "binaries_and_field": ("binaries_and_field", 0.5, {}, 1e-9),
    "triple": ("triple", 0.1, {}, 1e-9),
    "triple_M3": ("triple", 0.1, dict(M=3), 1e-9),
    "two_binaries_l1": ("two_binaries", 0.1, dict(l=1), 1e-9),
    "triple_l2_M2": ("triple", 0.1, dict(l=2, M=2, shell_ratio=1.6), 1e-9),
    "shared_view": ("shared_view", 0.1, {}, 1e-9),
    "global_view": ("global_view", 0.1, {}, 1e-9),
    "global_view_long": ("global_view", 0.5, {}, 1e-9),
    "backwards": ("two_binaries", -0.1, {}, 1e-9),
    "merge": ("binaries_and_field", 0.1, {}, 8e-4),
    "merge_shared_view": ("shared_view", 0.1, {}, 8e-4),
    "merge_global_view": ("global_view", 0.1, {}, 8e-4),
    "SI": ("triple", 0.1, dict(G=6.6743e-11, m0=MSUN), 1e-9),
    "slow_units": ("two_binaries", 0.1, dict(G=G * 2.0 ** -900), 1e-9),
}


def setup(name):
    kind, dt, kw, radius = CASES[name]
    x, v, m = system(kind)
    kw = dict(dt=dt, **kw)
    if name == "SI":
        x, v, m, radius, kw["dt"] = x * AU, v * AU / YR, m * MSUN, radius * AU, dt * YR
    if name == "slow_units":               # time in units of 2^450
        v, kw["dt"] = v * 2.0 ** -450, dt * 2.0 ** 450
    return x, v, m, np.full(len(m), radius), kw


@pytest.mark.parametrize("name", CASES)
def test_groups(orc, name):
    import paper_2304_07325_gb300 as sy
    from paper_2304_07325_gb300 import build

    build.build()
    x, v, m, radius, kw = setup(name)
    ref = orc.OracleSim(x, v, m, radius, params=orc.make_params(**kw))
    gpu = sy.System(x, v, m, radius, params=sy.default_params(**kw))
    for _ in range(2):
        twin = orc.OracleSim(x, v, ref.m, ref.radius, rhill=ref.rhill, params=orc.make_params(noise=1, **kw))
        twin.alive[...] = ref.alive
        twin.set_state(ref.x, ref.v)
        if not name.startswith("merge"):   # (a merged system goes on from its own state)
            gpu.set_state(ref.x, ref.v)
        assert ref.step(1) >= 0 and twin.step(1) >= 0
        gpu.step(1)
        assert gpu.sync() >= 0
        st = gpu.stats()
        calls = sum(ref.level_calls[1:])
        # the oracle takes the components of a level one by one, the group takes them together
        assert st.substeps <= calls + calls // 1000 and abs(st.max_depth - ref.max_depth_seen) <= 1
        if name.startswith("triple") or name == "SI":
            assert st.substeps >= calls - calls // 1000
        xg, _, mg, _, ag = gpu.get_state()
        assert np.array_equal(ag, ref.alive) and np.array_equal(mg, ref.m)
        live = ref.alive != 0
        norm = np.linalg.norm(ref.x, axis=1)
        rel = (np.linalg.norm(xg - ref.x, axis=1) / norm)[live]
        spread = (np.linalg.norm(twin.x - ref.x, axis=1) / norm)[live]
        assert np.all(rel <= np.maximum(1e-12, 100.0 * spread)), (rel, spread)
        if name.startswith("merge"):
            assert not live.all()
            break
    gpu.close()
