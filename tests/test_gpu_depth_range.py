"""Recursion levels at which the double-float arithmetic would leave FP32's range (needs a GB300): pairs of
point masses so close that r^-3 overflows, and pairs for which G m h^2 / 2, the factor of a kick in a run of
cleared sub-steps, underflows.  Against the oracle, over about a radian of mutual orbit or ten.

Bar: FP64 rounds x, near 1, to 2e-16 in every sub-step, which after N sub-steps is 2e-16 sqrt(N) phi / r of
the separation: 0.02 for r = 1e-13, N = 64, 0.02 for 4.4e-12, N = 1,024, phi = 10.  0.2 is ten times that;
a pair that feels no force, or a wrong one, is a radius and more from where it should be."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

G = 4.0 * math.pi ** 2


def circular_pair(r, n):
    """Two equal point masses on a circular mutual orbit of radius r and rate n, at 1 AU."""
    gm = 0.5 * n * n * r ** 3
    x = np.array([[1.0, 0.0, 0.0], [1.0, r, 0.0]])
    v = np.array([[0.0, 2.0 * math.pi, 0.0], [0.0, 2.0 * math.pi, 0.0]])
    v[0, 0] += 0.5 * n * r
    v[1, 0] -= 0.5 * n * r
    return x, v, np.full(2, gm / G)


# name: separation, rate, dt, R_0, deepest level, parameters
CASES = {
    "r3_overflows": (1e-13, 6.4e5, 2e-6, 1e-13 * 64.0 ** 2.5, 3, dict(shell_ratio=64.0)),
    "r3_overflows_M8": (1e-13, 6.4e5, 2e-6, 1e-13 * 64.0 ** 1.5, 2, dict(shell_ratio=64.0, M=8)),
    "kick_factor_underflows": (4.4e-12, 8.6e7, 2.0 ** -23, 2.82 * 4.4e-12, 5, dict(shell_ratio=1.26, max_depth=5)),
}


@pytest.mark.parametrize("third", [False, True], ids=["pair", "three"])
@pytest.mark.parametrize("name", CASES)
def test_against_the_oracle(orc, name, third):
    import paper_2304_07325_gb300 as sy
    from paper_2304_07325_gb300 import build

    build.build()
    r, n, dt, R0, depth, kw = CASES[name]
    tol = 0.2
    x, v, m = circular_pair(r, n)
    rh = np.full(2, R0 / 13.0)
    if third:                                # a third body that takes the pair through the levels of a group
        x = np.vstack([x, [1.0, -3.0 * r, 2.0 * r]])
        v = np.vstack([v, v.mean(0)])
        m, rh = np.append(m, 0.0), np.append(rh, rh[0])
    k = len(m)
    ref = orc.OracleSim(x, v, m, np.zeros(k), rhill=rh, params=orc.make_params(dt=dt, **kw))
    gpu = sy.System(x, v, m, np.zeros(k), rhill=rh, params=sy.default_params(dt=dt, **kw))
    assert ref.step(1) >= 0 and ref.max_depth_seen == depth
    gpu.step(1)
    assert gpu.sync() >= 0
    assert gpu.stats().max_depth == ref.max_depth_seen
    xg, vg = gpu.get_state()[:2]
    gpu.close()
    assert np.abs(xg - ref.x).max() <= 1e-12 and np.abs(vg - ref.v).max() <= max(1e-12, tol * n * r)
    dx, dr = xg[1] - xg[0], ref.x[1] - ref.x[0]
    dv, dw = vg[1] - vg[0], ref.v[1] - ref.v[0]
    # (the orbit has turned)
    assert np.linalg.norm(dr - (x[1] - x[0])) > r
    assert np.linalg.norm(dx - dr) <= tol * r, (dx, dr)
    assert np.linalg.norm(dv - dw) <= tol * n * r, (dv, dw)
