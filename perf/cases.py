"""Workloads this framework is timed on: what a user's program has it do, through its Python
entry points, from the smallest calls to the largest.

A "step" case is one turn of the loop an embedding program runs: hand the state over (set_state,
device arrays), advance it, wait, read the state back.  A "job" is a simulation from its start: set
the system up, advance it, read it back, give it back; its first step meets the pairs that fall
onto each other and merge, so it has the long chains of recursion sub-steps that a disk also meets
later on, which a step handed the same state again no longer has.  Either way every pass is the
same work.  Bodies that have left the system (merged or removed) carry no state: a program drops
them, so their positions and velocities are returned as zeros.

Sizes are those of the repository's configurations, tests and benchmark (the 1,000-, 5,000- and
10,000-body disks, 1,000 massive bodies with 100,000 field particles, batches of disks of uneven
size at the matched-accuracy step 0.125 yr) and ragged ones between them.  Inputs are the
synthetic planetesimal disks of paper_2304_07325_gb300/disk.py.
"""
import math

import numpy as np
import torch

import paper_2304_07325_gb300 as sy
from paper_2304_07325_gb300 import disk

PRECISION = {"fp64": sy.SYMBA_PRECISION_FP64, "mixed": sy.SYMBA_PRECISION_MIXED}


def _step(name, n, n_field=0, dt=0.5, precision="fp64", steps=1, M=4, spaced=False, rmin=0.0, rmax=0.0, kind="step"):
    c = {"kind": kind, "n": n, "n_field": n_field, "dt": dt, "precision": precision, "steps": steps, "M": M,
         "spaced": spaced, "rmin": rmin, "rmax": rmax}
    return dict(c, name=name) if name else c


def _batch(name, kind, disks, n_lo, n_hi, precision="mixed", dt=0.125):
    c = {"kind": kind, "disks": disks, "n_lo": n_lo, "n_hi": n_hi, "precision": precision, "dt": dt, "steps": 1}
    return dict(c, name=name) if name else c


def _energy(name, kind, n, n_field=0):
    c = {"kind": kind, "n": n, "n_field": n_field}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a hundred planets spaced by 5 mutual Hill radii (the accuracy run of the paper), ten
        # steps per call: hardly any arithmetic, so launches and latency count
        _step("hill_100", 100, dt=0.1, steps=10, spaced=True),
        # the 1,000-body parity disk: small kick, short chains of recursion sub-steps
        _step("disk_1000", 1000, steps=2),
        # the two benchmark disks, FP64 throughout, from their start
        _step("job_5000", 5000, kind="job"),
        _step("job_10000", 10000, kind="job"),
        # a ragged disk with the FP32-pair kick
        _step("job_7777_mixed", 7777, precision="mixed", kind="job"),
        # M = 3 (2.08 = 3^(2/3)) and bodies removed by distance: a run with ejections
        _step("disk_2500_M3_removal", 2500, M=3, rmin=1.0, rmax=25.0),
        # field-dominated disks: the massive/field rectangle, mixed at full size, FP64 ragged
        _step("job_1000_100000_mixed", 1000, n_field=100000, precision="mixed", kind="job"),
        _step("field_333_12345", 333, n_field=12345),
        # a parameter scan: uneven disks admitted to one pool, stepped by shared launches, read and
        # evicted, and disks as contexts that advance without waiting for one another
        _batch("pool_12_mixed", "pool", 12, 500, 4000),
        _batch("many_12", "many", 12, 1000, 5000, precision="fp64"),
        # the energy diagnostic of a run, and its allocation-free form on a program's own arrays
        _energy("energy_10000", "energy", 10000),
        _energy("energy_static_1500", "static", 1500, n_field=500),
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "job", "job", "field", "field", "pool", "many", "energy", "static"])
    precision = rng.choice(["fp64", "mixed"])
    if kind in ("step", "job"):
        dt = rng.choice([0.5, 0.5, 0.125, 0.1])
        n = logu(50, 9000)
        M = rng.choice([4, 4, 4, 3])
        rmin, rmax = rng.choice([(0.0, 0.0), (0.0, 0.0), (1.0, 30.0)])
        return _step("", n, dt=dt, precision=precision, steps=2 if kind == "step" and n <= 1000 else 1, M=M, rmin=rmin, rmax=rmax, kind=kind)
    if kind == "field":
        return _step("", logu(50, 1000), n_field=logu(1000, 60000), precision=precision, kind=rng.choice(["step", "job"]))
    if kind in ("pool", "many"):
        lo = logu(100, 1000)
        return _batch("", kind, rng.randint(2, 12), lo, lo * rng.randint(2, 4), precision=precision,
                      dt=rng.choice([0.125, 0.1]))
    return _energy("", kind, logu(30, 9000), n_field=rng.choice([0, 0, logu(100, 5000)]))


def _disk(case, seed):
    if case.get("spaced"):
        return disk.hill_spaced_disk(case["n"], seed=seed)
    return disk.planetesimal_disk(case["n"], seed, n_field=case.get("n_field", 0))


def _sizes(case):
    return disk.batch_sizes(case["disks"], 2000, case["n_lo"], case["n_hi"])


def _params(case):
    return sy.default_params(dt=case["dt"], M=case.get("M", 4), precision=PRECISION[case["precision"]],
                             rmin=case.get("rmin", 0.0), rmax=case.get("rmax", 0.0))


def _system(case, d):
    return sy.System(d.x, d.v, d.m, d.radius, n_massive=d.n_massive, params=_params(case))


def _on_gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _arrays(d):
    """A system's input arrays on the device: heliocentric state, masses, radii."""
    return [_on_gpu(a) for a in (d.x, d.v, d.m, d.radius)]


def prepare(case, seed):
    seed = 1 + seed % (1 << 30)
    kind = case["kind"]
    if kind == "step":
        s = _system(case, _disk(case, seed))
        x, v = s.get_state()[:2]
        return {"case": case, "sys": s, "x": _on_gpu(x), "v": _on_gpu(v)}
    if kind == "job":
        d = _disk(case, seed)
        return {"case": case, "in": _arrays(d), "nm": d.n_massive, "params": _params(case)}
    if kind in ("pool", "many"):
        ds = [disk.planetesimal_disk(n, seed + k) for k, n in enumerate(_sizes(case))]
        if kind == "many":
            ss = [_system(case, d) for d in ds]
            start = [s.get_state()[:2] for s in ss]
            return {"case": case, "sys": ss, "start": [(_on_gpu(x), _on_gpu(v)) for x, v in start]}
        tiles = sum(((d.n + 31) // 32) * ((d.n + 31) // 32 + 1) // 2 for d in ds)
        pool = sy.Pool(len(ds), sum(d.n for d in ds), tiles, PRECISION[case["precision"]])
        return {"case": case, "pool": pool, "in": [_arrays(d) for d in ds], "params": _params(case)}
    d = _disk(case, seed)
    if kind == "energy":
        return {"case": case, "sys": sy.System(d.x, d.v, d.m, d.radius, n_massive=d.n_massive)}
    s = sy.System(d.x, d.v, d.m, d.radius, n_massive=d.n_massive)
    x, v, m = s.get_state()[:3]
    return {"case": case, "nm": d.n_massive, "x": _on_gpu(x), "v": _on_gpu(v), "m": _on_gpu(m),
            "out": torch.zeros(4, dtype=torch.float64, device="cuda")}


def _live(states):
    """The states of one or several systems, end to end, without the bodies that have left."""
    x, v, m, r, a = (np.concatenate(t) for t in zip(*states))
    keep = (a != 0)[:, None]
    return {"x": np.where(keep, x, 0.0), "v": np.where(keep, v, 0.0), "m": m, "radius": r, "alive": a}


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "step":
        s = state["sys"]
        s.set_state(state["x"], state["v"])
        s.step(case["steps"])
        s.sync()
        return _live([s.get_state()])
    if kind == "job":
        s = sy.System(*state["in"], n_massive=state["nm"], params=state["params"])
        s.step(case["steps"])
        s.sync()
        out = s.get_state()
        s.close()
        return _live([out])
    if kind == "pool":
        pool = state["pool"]
        slots = [pool.admit(*a, params=state["params"]) for a in state["in"]]
        pool.step(case["steps"])
        pool.sync()
        out = [pool.get_state(k) for k in slots]
        for k in slots:
            pool.evict(k)
        return _live(out)
    if kind == "many":
        for s, (x, v) in zip(state["sys"], state["start"]):
            s.set_state(x, v)
        sy.step_many(state["sys"], case["steps"])
        return _live([s.get_state() for s in state["sys"]])
    if kind == "energy":
        E, L = state["sys"].energy()
        return {"E": E, "L": L}
    p = sy._ptr
    st = torch.cuda.current_stream()
    sy._check(sy.lib().symba_energy_static(state["x"].shape[0], state["nm"], p(state["x"]), p(state["v"]), p(state["m"]),
                                           sy.G_default(), 1.0, p(state["out"]), sy._stream_handle(st)),
              "symba_energy_static")
    return state["out"]


def work(case):
    kind = case["kind"]
    if kind in ("pool", "many"):
        sizes = _sizes(case)
        n, pairs = sum(sizes), sum(k * (k - 1) // 2 for k in sizes)
    else:
        nm, nf = case["n"], case["n_field"]
        n, pairs = nm + nf, nm * (nm - 1) // 2 + nm * nf
    if kind in ("energy", "static"):
        # positions, velocities and masses in; per pair 3 differences, r^2, root, quotient, sum
        return {"bytes": 56.0 * n + 32.0, "flops": 13.0 * pairs + 40.0 * n}
    # state in and out (x, v; m, radius, flags out); per pair two kicks of 26 and the encounter
    # check of 18; per body a Kepler drift of about 300; the recursion's sub-steps, which depend
    # on the encounters a disk has, are left out
    return {"bytes": n * (48.0 + 68.0), "flops": case["steps"] * (70.0 * pairs + 300.0 * n)}


# ---------------------------------------------------------------------------------------------
# the same results from plain numpy and Python floats in 64 bits
# ---------------------------------------------------------------------------------------------
class _TooLong(Exception):
    pass


_CUT = 150000        # recursion sub-steps of one exact() at most (some tens of microseconds each)


def _f3(x):
    return 0.0 if x <= 0.0 else 1.0 if x >= 1.0 else x ** 4 * (35.0 + x * (-84.0 + x * (70.0 - 20.0 * x)))


def _met(dx, dv, R, h):
    """Whether the straight-line relative motion comes closer than R within [0, h]."""
    r2 = dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2]
    if r2 < R * R:
        return True
    vr = dx[0] * dv[0] + dx[1] * dv[1] + dx[2] * dv[2]
    if vr >= 0.0:
        return False
    v2 = dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]
    t = -vr / v2
    if t < h:
        return r2 - vr * vr / v2 < R * R
    return r2 + h * (2.0 * vr + h * v2) < R * R


def _kepler(mu, h, x, v):
    """Two-body motion over h (elliptic orbits; the disks have no others)."""
    r0 = math.sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2])
    v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2]
    u = x[0] * v[0] + x[1] * v[1] + x[2] * v[2]
    a = 1.0 / (2.0 / r0 - v2 / mu)
    if not a > 0.0:
        raise _TooLong
    n = math.sqrt(mu / a) / a
    ec, es, M = 1.0 - r0 / a, u / (n * a * a), n * h
    X = M
    for _ in range(60):
        s, om = math.sin(X), 2.0 * math.sin(0.5 * X) ** 2
        d = -(X - ec * s + es * om - M) / (1.0 - ec * (1.0 - om) + es * s)
        X += d
        if abs(d) <= 1e-15 * max(1e-30, abs(X)):
            break
    s, om = math.sin(X), 2.0 * math.sin(0.5 * X) ** 2
    if abs(X) < 0.5:
        z, t, xs = X * X, X ** 3 / 6.0, 0.0
        for k in range(2, 12):
            xs += t
            t *= -z / (2 * k * (2 * k + 1))
    else:
        xs = X - s
    r = a * (1.0 - ec * (1.0 - om) + es * s)
    f, g = -(a / r0) * om, h - xs / n
    fd, gd = -(a * a * n * s) / (r * r0), -(a / r) * om
    return ([x[k] + (f * x[k] + g * v[k]) for k in range(3)], [v[k] + (fd * x[k] + gd * v[k]) for k in range(3)])


class _Sim:
    def __init__(self, d, dt, M, rmin, rmax):
        self.G, self.m0, self.lam, self.dt, self.M, self.rmin, self.rmax = 4.0 * math.pi ** 2, 1.0, 6.5, dt, M, rmin, rmax
        self.nm, self.x, self.m, self.R = d.n_massive, d.x.copy(), d.m.copy(), d.radius.copy()
        q = np.array([math.fsum(self.m * d.v[:, c]) for c in range(3)]) / (self.m0 + math.fsum(self.m))
        self.v = d.v - q
        r = np.sqrt((d.x ** 2).sum(1))
        inv = 2.0 / r - (d.v ** 2).sum(1) / (self.G * (self.m0 + self.m))
        a = np.where(inv > 0.0, 1.0 / np.where(inv > 0.0, inv, 1.0), r)
        self.rh = a * np.cbrt(self.m / (3.0 * self.m0))
        self.alive = np.ones(len(self.m), dtype=np.int32)
        self.c = [2.08 ** -k for k in range(40)]
        self.subs = 0

    def sun(self):
        h, on = 0.5 * self.dt, self.alive != 0
        P = np.array([math.fsum((self.m * self.v[:, c])[on]) for c in range(3)])
        self.x[on] += h * (P / self.m0)

    def check(self):
        """The pairs that meet within the step, as a set of (i, j), i < j."""
        pairs, on = set(), self.alive != 0
        for i in range(self.nm):
            if not on[i]:
                continue
            js = np.arange(i + 1, len(self.m))
            dx, dv = self.x[js] - self.x[i], self.v[js] - self.v[i]
            R = self.lam * (self.rh[i] + self.rh[js])
            near = np.sqrt((dx ** 2).sum(1)) - abs(self.dt) * np.sqrt((dv ** 2).sum(1)) <= R * (1.0 + 1e-9) + 1e-9
            for j in js[near & on[js]]:
                if _met(self.x[j] - self.x[i], self.v[j] - self.v[i], self.lam * (self.rh[i] + self.rh[j]), self.dt):
                    pairs.add((i, int(j)))
        return sorted(pairs)

    def weight(self, R0, r, k):
        def g(j):
            return _f3((r - R0 * self.c[j + 1]) / (R0 * self.c[j] - R0 * self.c[j + 1])) if j >= 0 else 0.0
        return g(k) - g(k - 1)

    def kick(self, pairs):
        a = np.zeros_like(self.x)
        gm, n = self.G * self.m * (self.alive != 0), len(self.m)
        for i in range(self.nm):
            if not self.alive[i]:
                continue
            d = self.x[i + 1:n] - self.x[i]
            r2 = (d ** 2).sum(1)
            q = np.where(self.alive[i + 1:n] != 0, 1.0 / (r2 * np.sqrt(r2)), 0.0)
            a[i] += ((gm[i + 1:n] * q)[:, None] * d).sum(0)
            a[i + 1:n] -= (gm[i] * q)[:, None] * d
        for i, j in pairs:
            if self.alive[i] and self.alive[j]:
                d = self.x[j] - self.x[i]
                r = math.sqrt((d ** 2).sum())
                w = self.weight(self.lam * (self.rh[i] + self.rh[j]), r, 0) - 1.0
                a[i] += w * gm[j] / r ** 3 * d
                a[j] -= w * gm[i] / r ** 3 * d
        on = self.alive != 0
        self.v[on] += 0.5 * self.dt * a[on]

    def merge(self, X, V, i, j):
        mi, mj = self.m[i], self.m[j]
        if mi + mj > 0.0:
            X[i] = [(mi * X[i][k] + mj * X[j][k]) / (mi + mj) for k in range(3)]
            V[i] = [(mi * V[i][k] + mj * V[j][k]) / (mi + mj) for k in range(3)]
        self.R[i] = (self.R[i] ** 3 + self.R[j] ** 3) ** (1.0 / 3.0)
        if mi > 0.0:
            self.rh[i] *= ((mi + mj) / mi) ** (1.0 / 3.0)
        self.m[i] = mi + mj
        self.m[j] = self.R[j] = self.rh[j] = 0.0
        self.alive[j] = 0

    def encounter(self, X, V, pairs, k, h):
        """E_k over h for the pairs of F_{k-1}; X, V: positions and velocities of their bodies."""
        self.subs += 1
        if self.subs > _CUT or k > 20:
            raise _TooLong
        deep = []
        for i, j in pairs:
            if not (self.alive[i] and self.alive[j]):
                continue
            dx = [X[j][c] - X[i][c] for c in range(3)]
            Rc = self.R[i] + self.R[j]
            if dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2] < Rc * Rc:
                self.merge(X, V, i, j)
            elif _met(dx, [V[j][c] - V[i][c] for c in range(3)], self.lam * (self.rh[i] + self.rh[j]) * self.c[k], h):
                deep.append((i, j))
        self.pull(X, V, pairs, k, 0.5 * h)
        inside = {b for p in deep for b in p}
        for b in {b for p in pairs for b in p}:
            if b not in inside and self.alive[b]:
                X[b], V[b] = _kepler(self.G * self.m0, h, X[b], V[b])
        if deep:
            for _ in range(self.M):
                self.encounter(X, V, deep, k + 1, h / self.M)
        self.pull(X, V, pairs, k, 0.5 * h)

    def pull(self, X, V, pairs, k, hh):
        for i, j in pairs:
            if self.alive[i] and self.alive[j]:
                d = [X[j][c] - X[i][c] for c in range(3)]
                r = math.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
                w = self.weight(self.lam * (self.rh[i] + self.rh[j]), r, k) * hh * self.G / r ** 3
                wi, wj = w * self.m[j], w * self.m[i]
                V[i] = [V[i][c] + wi * d[c] for c in range(3)]
                V[j] = [V[j][c] - wj * d[c] for c in range(3)]

    def step(self):
        self.sun()
        pairs = self.check()
        self.kick(pairs)
        root = {b: b for p in pairs for b in p}

        def find(b):
            while root[b] != b:
                b = root[b]
            return b

        for i, j in pairs:
            a, b = sorted((find(i), find(j)))
            root[b] = a
        groups = {}
        for p in pairs:
            groups.setdefault(find(p[0]), []).append(p)
        for b in np.nonzero(self.alive)[0]:
            if int(b) not in root:
                self.x[b], self.v[b] = _kepler(self.G * self.m0, self.dt, self.x[b].tolist(), self.v[b].tolist())
        for ps in groups.values():
            X = {b: self.x[b].tolist() for p in ps for b in p}
            V = {b: self.v[b].tolist() for p in ps for b in p}
            for _ in range(self.M):
                self.encounter(X, V, ps, 1, self.dt / self.M)
            for b in X:
                self.x[b], self.v[b] = X[b], V[b]
        self.kick(pairs)
        r2 = (self.x ** 2).sum(1)
        out = (self.alive != 0) & ((self.rmin > 0.0) & (r2 < self.rmin ** 2) | (self.rmax > 0.0) & (r2 > self.rmax ** 2))
        self.m[out] = self.R[out] = self.rh[out] = 0.0
        self.alive[out] = 0
        self.sun()


def _exact_energy(d):
    G, n = 4.0 * math.pi ** 2, len(d.m)
    q = np.array([math.fsum(d.m * d.v[:, c]) for c in range(3)]) / (1.0 + math.fsum(d.m))
    v = d.v - q
    P = [math.fsum(d.m * v[:, c]) for c in range(3)]
    terms = [0.5 * d.m * (v ** 2).sum(1), -G * d.m / np.sqrt((d.x ** 2).sum(1)), [0.5 * (P[0] ** 2 + P[1] ** 2 + P[2] ** 2)]]
    for i in range(min(d.n_massive, n - 1)):
        r = np.sqrt(((d.x[i + 1:] - d.x[i]) ** 2).sum(1))
        terms.append([-G * d.m[i] * math.fsum(d.m[i + 1:] / r)])
    L = np.cross(d.x, v) * d.m[:, None]
    return math.fsum(t for part in terms for t in part), np.array([math.fsum(L[:, c]) for c in range(3)])


def exact(case, seed):
    seed = 1 + seed % (1 << 30)
    kind = case["kind"]
    if kind in ("energy", "static"):
        E, L = _exact_energy(_disk(case, seed))
        return {"E": E, "L": L} if kind == "energy" else np.concatenate([[E], L])
    if kind in ("pool", "many"):
        sims = [_Sim(disk.planetesimal_disk(n, seed + k), case["dt"], 4, 0.0, 0.0)
                for k, n in enumerate(_sizes(case)) if n <= 2000]
        if len(sims) < case["disks"]:
            return None
    else:
        if case["n"] > 3000 or case["n"] * (case["n"] + case["n_field"]) > 20_000_000:
            return None
        sims = [_Sim(_disk(case, seed), case["dt"], case["M"], case["rmin"], case["rmax"])]
    try:
        for s in sims:
            for _ in range(case["steps"]):
                s.step()
    except _TooLong:
        return None
    got = _live([(s.x, s.v, s.m, s.R, s.alive) for s in sims])
    return {k: got[k] for k in ("x", "v", "m", "radius", "alive")}
