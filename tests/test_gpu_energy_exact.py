"""Energy and angular momentum as the correctly rounded sums of their terms (needs a GB300), against
math.fsum over numpy's terms in the same operation order: equality of every bit, on the pair terms'
integer arithmetic and its way out (terms outside the 2^50 range of a warp's sum, massless bodies,
subnormal products), at the edges of tiles and strips."""
import ctypes
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_2304_07325_gb300 import disk  # noqa: E402

M0 = 1.0


def _exact(x, v, m, nm, G):
    n = len(m)
    v2 = v[:, 0] * v[:, 0] + v[:, 1] * v[:, 1] + v[:, 2] * v[:, 2]
    r = np.sqrt(x[:, 0] * x[:, 0] + x[:, 1] * x[:, 1] + x[:, 2] * x[:, 2])
    P = [math.fsum(m * v[:, c]) for c in range(3)]
    terms = [(0.5 * m) * v2, -((G * M0) * m) / r, np.array([(P[0] * P[0] + P[1] * P[1] + P[2] * P[2]) / (2.0 * M0)])]
    for i in range(min(nm, n - 1)):
        d = x[i + 1:] - x[i]
        s = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2]
        terms.append(-((G * m[i]) * m[i + 1:]) / np.sqrt(s))
    L = [m * (x[:, a] * v[:, b] - x[:, b] * v[:, a]) for a, b in ((1, 2), (2, 0), (0, 1))]
    return math.fsum(np.concatenate(terms)), [math.fsum(t) for t in L]


def _state(n, nf, what):
    d = disk.planetesimal_disk(n, 300 + n, n_field=nf)
    x, v, m = d.x.copy(), d.v.copy(), d.m.copy()
    rng = np.random.default_rng(n + nf)
    if what == "massless":
        m[rng.random(n + nf) < 0.4] = 0.0
    elif what == "wide":                 # terms over 2^140: most of them outside any one window
        m *= 2.0 ** rng.integers(-40, 41, n + nf)
        x *= 2.0 ** rng.integers(-30, 31, (n + nf, 1))
    elif what == "subnormal":            # G m_i m_j below and around 2^-1022
        m = 2.0 ** -(500.0 + rng.integers(0, 40, n + nf)) * (1.0 + rng.random(n + nf))
    elif what == "squares":              # exact roots, and roots next to a rounding boundary
        x = np.round(x * 64.0) / 64.0
        x[:, 2] = 0.0
        x[: n // 2, 1] = 0.0
        x += np.arange(n + nf)[:, None] * np.array([[1.0, 0.0, 0.0]])
    return x, v, m


@pytest.mark.parametrize("n,nf,what", [(1, 0, "disk"), (2, 0, "disk"), (31, 2, "disk"), (33, 0, "disk"), (64, 65, "disk"),
                                       (300, 411, "disk"), (1300, 0, "disk"), (90, 50, "massless"), (150, 90, "wide"),
                                       (70, 30, "subnormal"), (200, 100, "squares")])
def test_sums_and_terms_to_the_last_bit(n, nf, what):
    import torch

    import paper_2304_07325_gb300 as sy
    from paper_2304_07325_gb300 import build

    build.build()
    x, v, m = _state(n, nf, what)
    G = sy.default_params().G
    E, L = _exact(x, v, m, n, G)
    t = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (x, v, m)]
    out = torch.full((4,), math.nan, dtype=torch.float64, device="cuda")
    ptr = lambda a: ctypes.c_void_p(a.data_ptr())
    assert sy.lib().symba_energy_static(n + nf, n, ptr(t[0]), ptr(t[1]), ptr(t[2]), G, M0, ptr(out), None) == sy.SYMBA_OK
    torch.cuda.synchronize()
    assert out.tolist() == [E] + L
    if what == "subnormal":              # no Hill radii for such masses
        return
    s = sy.System(x, v, m, np.zeros(n + nf), n_massive=n, params=sy.default_params(m0=M0))
    xs, vs, ms = s.get_state()[:3]
    E, L = _exact(xs, vs, ms, n, G)
    Eg, Lg = s.energy()
    assert [Eg] + list(Lg) == [E] + L
    s.close()
