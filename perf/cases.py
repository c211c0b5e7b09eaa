"""What a user of this library has it do, as cases to measure.

A case is one call (or one short run) through the Python binding: a force
solve of one system in the FP64 or the mixed form, at order 3 or above, from
device or host arrays, launched by the host or replayed as one graph; a forest
of systems; a short leapfrog integration; a solve with the learned pair
selector; exact direct sums.

``exact`` evaluates the same method in plain PyTorch float64 (its own tree,
walk, expansions and sums, written from the method's formulas).
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1706_06989_gb300 import fmm, ics, selector

_DEFAULT = dict(kind="solve", ics="plummer", n=0, theta=0.5, n_crit=25, variant="TC", precision="fp64", order=3,
                eps=0.0, graph=False)


def _case(**kw):
    return {**_DEFAULT, **kw}


def listed():
    return [
        # the smallest system of the tests and the smoke check: one solve of a
        # few thousand bodies inside a host loop, all latency and launches
        _case(name="plummer_2000_fp64", n=2000),
        # a mid-sized system solved again and again as one graph launch (the
        # mode for repeated solves of the same buffers)
        _case(name="plummer_65536_mixed_graph", n=65536, precision="mixed", graph=True),
        # an odd-sized run of the paper's own test problem, coarse angle, no
        # correction: the cheap end of the theta sweep
        _case(name="dwd_250007_uc_theta0.8", ics="dwd", n=250007, theta=0.8, variant="UC"),
        # end to end from host memory (the bodies come from and go back to the
        # caller's arrays), torque correction by Eq. 8
        _case(name="plummer_262144_host_tco", kind="host", n=262144, variant="TCO"),
        # the benchmark's workload in both forms
        _case(name="plummer_1048576_fp64", n=1048576),
        _case(name="plummer_1048576_mixed", n=1048576, precision="mixed"),
        # the largest: a halo with a thin disc and a mass spectrum, the shape of
        # a galaxy model
        _case(name="disc_4194304_mixed", ics="disc_spectrum", n=4194304, precision="mixed"),
        # higher order of App. A (generated code at 4 and 5, tables from 6)
        _case(name="plummer_65536_order5", n=65536, order=5),
        _case(name="plummer_16384_order6", n=16384, order=6, theta=0.7),
        # many small independent systems solved together
        _case(name="forest_48_mixed", kind="forest", n=48, n_crit=32, precision="mixed"),
        # a few steps of a softened binary, state and conserved totals returned
        _case(name="binary_200000_leapfrog", kind="leapfrog", ics="binary", n=200000, precision="mixed", eps=1e-3),
        # the learned pair selector with the committed network
        _case(name="disc_262144_selector", kind="selector", ics="disc_spectrum", n=262144, theta=0.45,
              precision="mixed"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | (1 if rng.random() < 0.5 else 0)

    which = rng.random()
    variant = rng.choice(["UC", "TC", "TC", "TCO"])
    theta = round(rng.uniform(0.4, 1.0), 3)
    n_crit = rng.choice([8, 16, 25, 25, 32, 48])
    system = rng.choice(["plummer", "dwd", "disc", "disc_spectrum", "binary", "cube"])
    precision = rng.choice(["fp64", "mixed"])
    if which < 0.10:
        return _case(kind="forest", n=rng.randrange(2, 40), theta=max(theta, 0.5), n_crit=n_crit, variant=variant,
                     precision=precision)
    if which < 0.20:
        return _case(kind="leapfrog", ics="binary", n=size(2000, 300000), theta=max(theta, 0.5), precision=precision,
                     variant=rng.choice(["UC", "TC"]), eps=rng.choice([1e-3, 2e-3, 5e-3]))
    if which < 0.35:
        order = rng.choice([4, 4, 5, 5, 6, 7])
        return _case(ics=system, n=size(1000, 100000 if order < 6 else 12000), theta=max(theta, 0.6), order=order,
                     n_crit=max(n_crit, 16))
    return _case(kind="host" if rng.random() < 0.2 else "solve", ics=system, n=size(1500, 1000000), theta=theta,
                 n_crit=n_crit, variant=variant, precision=precision, graph=rng.random() < 0.2,
                 eps=rng.choice([0.0, 0.0, 0.0, 1e-3]))


LEAP_STEPS, FOREST_MIN, FOREST_MAX = 4, 1024, 16384


def _system(case, seed):
    n = case["n"]
    if case["ics"] == "dwd":
        return ics.dwd(n, seed=seed)
    if case["ics"] == "disc":
        return ics.hernquist_disc(n, seed=seed)
    if case["ics"] == "disc_spectrum":
        return ics.hernquist_disc(n, seed=seed, mass_spectrum=True)
    if case["ics"] == "binary":
        return ics.binary_plummer(n, seed=seed)
    if case["ics"] == "cube":
        return ics.uniform_cube(n, seed=seed, mass_spread=True)
    return ics.plummer(n, seed=seed)


def _forest(case, seed):
    """Plummer spheres of log-uniform sizes (the same sizes for every seed);
    (offsets, bodies)."""
    sizes = ics.ensemble_sizes(case["n"], seed=case["n"], nmin=FOREST_MIN, nmax=FOREST_MAX)
    parts = [ics.plummer(int(s), seed=seed + 1 + k) for k, s in enumerate(sizes)]
    cat = lambda f: np.concatenate([getattr(p, f) for p in parts])  # noqa: E731
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64), ics.Bodies(cat("x"), cat("y"), cat("z"), cat("m"))


def _timestep():
    # a thousandth of the orbit of the binary (masses 0.6 and 0.9, separation 1)
    return 2.0 * math.pi / math.sqrt(1.5) / 1000.0


def prepare(case, seed):
    dev = torch.device("cuda")
    offsets = None
    if case["kind"] == "forest":
        offsets, b = _forest(case, seed)
    else:
        b = _system(case, seed)
    s = fmm.FMM(theta=case["theta"], n_crit=case["n_crit"], variant=case["variant"], precision=case["precision"],
                order_P=case["order"])
    if case["eps"]:
        s.set_softening(case["eps"])
    if case["graph"]:
        s.set_graph(True)
    state = {"case": case, "solver": s, "offsets": offsets}
    if case["kind"] == "host":
        # pinned arrays, as a program that streams bodies through the GPU keeps
        state["bodies"] = [torch.from_numpy(v).pin_memory() for v in (b.x, b.y, b.z, b.m)]
        state["out"] = [torch.empty(b.n, dtype=torch.float64).pin_memory() for _ in range(3)]
        return state
    state["bodies"] = [torch.from_numpy(v).to(dev) for v in (b.x, b.y, b.z, b.m)]
    state["out"] = tuple(torch.empty(b.n, dtype=torch.float64, device=dev) for _ in range(3))
    if case["kind"] == "leapfrog":
        state["start"] = [torch.from_numpy(v).to(dev) for v in (b.x, b.y, b.z, b.vx, b.vy, b.vz)]
    if case["kind"] == "selector":
        p = selector.trained_params()
        s.selector_set(p["params"], p["log10_target"], theta_max=p["theta_max"], min_work=p["min_work"],
                       rule=p["rule"])
    return state


def run(state):
    case, s = state["case"], state["solver"]
    if case["kind"] == "host":
        return list(s.solve_host(*state["bodies"], out=state["out"]))
    if case["kind"] == "forest":
        return list(s.solve_batch(*state["bodies"], state["offsets"], out=state["out"]))
    if case["kind"] == "leapfrog":
        q = [v.clone() for v in state["start"]]
        acc, mom = s.leapfrog(*q, state["bodies"][3], _timestep(), LEAP_STEPS, acc=state["out"])
        return {"state": q, "acc": list(acc), "mom": mom}
    return list(s.solve(*state["bodies"], out=state["out"]))


def _interactions(n, case):
    """Typical counts of a solve: accepted cell pairs and mutual body pairs."""
    angle = (0.5 / case["theta"]) ** 3
    near = min(n * (n - 1) / 2.0, 16.0 * case["n_crit"] * angle * n)
    far = min(1.0, n / 20000.0) * 24.0 * (25.0 / case["n_crit"]) * angle * n
    return far, near


def work(case):
    if case["kind"] == "forest":
        sizes = [math.sqrt(FOREST_MIN * FOREST_MAX)] * case["n"]
    else:
        sizes = [case["n"]]
    solves = LEAP_STEPS + 1 if case["kind"] == "leapfrog" else 1
    P = case["order"]
    terms = math.comb(P + 3, 3)
    per_pair = (235.0 if case["variant"] != "UC" else 162.0) if P == 3 else 2.0 * terms * terms
    flops = sum(far * per_pair + 25.0 * near for far, near in (_interactions(n, case) for n in sizes))
    n = sum(sizes)
    # bodies in, accelerations out; a leapfrog run also reads and writes its state
    words = 7 + (12 if case["kind"] == "leapfrog" else 0)
    return {"bytes": 8.0 * words * n, "flops": flops * solves}


# --------------------------------------------------------------------------
# the method in plain PyTorch float64
# --------------------------------------------------------------------------

def _multi_indices(order):
    return [(a, b, n - a - b) for n in range(order + 1) for a in range(n, -1, -1) for b in range(n - a, -1, -1)]


def _plus(a, b):
    return tuple(i + j for i, j in zip(a, b))


def _unit(k):
    return tuple(int(i == k) for i in range(3))


def _factorial(a):
    return math.prod(math.factorial(i) for i in a)


def _powers(x, order):
    """{a: x^a} for |a| <= order, x = three tensors."""
    out = {(0, 0, 0): torch.ones_like(x[0])}
    for a in _multi_indices(order)[1:]:
        k = next(i for i in range(3) if a[i])
        out[a] = out[tuple(v - (i == k) for i, v in enumerate(a))] * x[k]
    return out


def _derivatives(r, eps2, order):
    """{a: d^a G} of G = -1/sqrt(r.r + eps2), |a| <= order, from the Leibniz
    expansion of d^k [R^2 d_i G + r_i G] = 0."""
    R2 = r[0] ** 2 + r[1] ** 2 + r[2] ** 2 + eps2
    inv = 1.0 / R2
    D = {(0, 0, 0): -R2.rsqrt()}
    get = lambda a: D[a] if min(a) >= 0 else None  # noqa: E731
    for a in _multi_indices(order)[1:]:
        i = max(range(3), key=lambda j: a[j])
        k = tuple(v - (j == i) for j, v in enumerate(a))
        s = r[i] * D[k]
        below = get(tuple(v - (j == i) for j, v in enumerate(k)))
        if below is not None:
            s = s + k[i] * below
        for j in range(3):
            if k[j] >= 1:
                s = s + 2 * k[j] * r[j] * D[tuple(v - (q == j) for q, v in enumerate(a))]
            if k[j] >= 2:
                s = s + k[j] * (k[j] - 1) * D[tuple(v - 2 * (q == j) for q, v in enumerate(a))]
        D[a] = -s * inv
    return D


class _Tree:
    """Octree over 63-bit Morton keys: a cell of at most n_crit bodies, or of
    level 21, is a leaf; cells are numbered breadth first."""

    def __init__(self, x, m, n_crit, order):
        dev, n = m.device, m.shape[0]
        lo = [v.min() for v in x]
        ext = max(float(v.max() - l) for v, l in zip(x, lo))
        scale = 2.0 ** 21 / ext if ext > 0 else 0.0
        key = torch.zeros(n, dtype=torch.int64, device=dev)
        for d in range(3):
            q = ((x[d] - lo[d]) * scale).floor().clamp(max=2.0 ** 21 - 1).to(torch.int64)
            for b in range(21):
                key |= ((q >> b) & 1) << (3 * b + d)
        self.order = torch.argsort(key, stable=True)
        key, self.x, self.m = key[self.order], [v[self.order] for v in x], m[self.order]
        body = torch.arange(n, device=dev)
        begin, count, level, first, nchild, self.levels = [], [], [], [], [], []
        b0, c0 = torch.zeros(1, dtype=torch.int64, device=dev), torch.full((1,), n, dtype=torch.int64, device=dev)
        base = 0
        for l in range(22):
            k = b0.shape[0]
            self.levels.append((base, base + k))
            split = (c0 > n_crit) & (l < 21)
            begin.append(b0), count.append(c0), level.append(torch.full_like(b0, l))
            f, nc = torch.zeros_like(b0), torch.zeros_like(b0)
            sb, sc = b0[split], c0[split]
            if sb.shape[0] == 0:
                first.append(f), nchild.append(nc)
                break
            prefix = key >> (3 * (20 - l))
            edge = torch.ones(n, dtype=torch.bool, device=dev)
            edge[1:] = prefix[1:] != prefix[:-1]
            own = torch.searchsorted(sb, body, right=True) - 1
            inside = (own >= 0) & (body < (sb + sc)[own.clamp(min=0)])
            edge[sb] = True
            nb = torch.nonzero(edge & inside).flatten()
            par = own[nb]
            nxt = torch.cat([nb[1:], nb.new_full((1,), n)])
            kids = torch.bincount(par, minlength=sb.shape[0])
            nc[split] = kids
            f[split] = base + k + torch.cumsum(kids, 0) - kids
            first.append(f), nchild.append(nc)
            base += k
            b0, c0 = nb, torch.minimum(nxt, (sb + sc)[par]) - nb
        cat = torch.cat
        self.begin, self.count, self.level, self.first, self.nchild = (
            cat(begin), cat(count), cat(level), cat(first), cat(nchild))
        self.leaf = self.nchild == 0
        C = self.begin.shape[0]
        self.C, self.idx = C, _multi_indices(order)
        self.M = torch.zeros(C, dtype=torch.float64, device=dev)
        self.Z = [torch.zeros_like(self.M) for _ in range(3)]
        self.R = torch.zeros_like(self.M)
        self.mom = {a: torch.zeros_like(self.M) for a in self.idx}
        for lo_, hi_ in self.levels:
            cell, at = self.bodies(torch.arange(lo_, hi_, device=dev))
            mu, p = self.m[at], [v[at] for v in self.x]
            self.M.index_add_(0, cell, mu)
            for d in range(3):
                self.Z[d].index_add_(0, cell, mu * p[d])
                self.Z[d][lo_:hi_] /= self.M[lo_:hi_]
            off = [p[d] - self.Z[d][cell] for d in range(3)]
            self.R.scatter_reduce_(0, cell, (off[0] ** 2 + off[1] ** 2) + off[2] ** 2, "amax")
            for a, v in _powers(off, order).items():
                self.mom[a].index_add_(0, cell, mu * v)
        self.R = self.R.sqrt()

    def bodies(self, cells):
        """(cell, body) of every body of the given cells."""
        c = self.count[cells]
        cell = torch.repeat_interleave(cells, c)
        start = torch.repeat_interleave(self.begin[cells] - (torch.cumsum(c, 0) - c), c)
        return cell, start + torch.arange(cell.shape[0], device=cells.device)


def _walk(t, theta):
    """Accepted pairs and leaf pairs (self pairs among them) of the dual walk."""
    far, near = [], []
    A = torch.zeros(1, dtype=torch.int64, device=t.M.device)
    B = A.clone()
    ramp = lambda k: torch.arange(int(k.sum()), device=k.device) - torch.repeat_interleave(  # noqa: E731
        torch.cumsum(k, 0) - k, k)
    while A.shape[0]:
        same = A == B
        d2 = sum((z[A] - z[B]) ** 2 for z in t.Z)
        sep = ~same & (theta * theta * d2 >= (t.R[A] + t.R[B]) ** 2)
        leaves = ~sep & t.leaf[A] & t.leaf[B]
        far.append((A[sep], B[sep]))
        near.append((A[leaves], B[leaves]))
        s = same & ~leaves
        k = t.nchild[A[s]]
        own, j = torch.repeat_interleave(A[s], k * k), ramp(k * k)
        kk = t.nchild[own]
        u, v = j // kk, j % kk
        up = u <= v
        nA, nB = (t.first[own] + u)[up], (t.first[own] + v)[up]
        o = ~same & ~sep & ~leaves
        a, b = A[o], B[o]
        tie = t.R[a] == t.R[b]
        pick = torch.where(tie, (t.level[a] < t.level[b]) | ((t.level[a] == t.level[b]) & (a < b)), t.R[a] > t.R[b])
        pick = torch.where(t.leaf[a], torch.zeros_like(pick), torch.where(t.leaf[b], torch.ones_like(pick), pick))
        sp, ot = torch.where(pick, a, b), torch.where(pick, b, a)
        k = t.nchild[sp]
        A = torch.cat([nA, torch.repeat_interleave(t.first[sp], k) + ramp(k)])
        B = torch.cat([nB, torch.repeat_interleave(ot, k)])
    join = lambda lst: tuple(torch.cat([p[i] for p in lst]) for i in (0, 1))  # noqa: E731
    return join(far), join(near)


def _far_field(t, far, variant, P, eps2):
    """Local expansions {a: L^a}, 1 <= |a| <= P, of every cell: both sides of
    every accepted pair, each as the field of the source S in the target T."""
    L = {a: torch.zeros_like(t.M) for a in t.idx[1:]}
    step = (1 << 24) // math.comb(P + 4, 3)
    top = [a for a in t.idx if sum(a) == P]
    for T_, S_ in (far, far[::-1]):
        for at in range(0, T_.shape[0], step):
            T, S = T_[at:at + step], S_[at:at + step]
            r = [z[T] - z[S] for z in t.Z]
            D = _derivatives(r, eps2, P + 1)
            src = {b: t.mom[b][S] for b in t.idx if sum(b) != 1}  # dipoles about a centre of mass vanish
            for a in t.idx[1:]:
                v = sum((-1) ** sum(b) / _factorial(b) * src[b] * D[_plus(a, b)] for b in src if sum(a) + sum(b) <= P)
                L[a].index_add_(0, T, v)
            if variant == "UC":
                continue
            tgt = {b: t.mom[b][T] for b in src}
            if variant == "TCO":  # order 3, Eq. (8): the terms of D_ijkl without a factor r_i
                O = {a: src[a] * tgt[(0, 0, 0)] - tgt[a] * src[(0, 0, 0)] for a in top}
                R2 = r[0] ** 2 + r[1] ** 2 + r[2] ** 2 + eps2
                F = []
                for i in range(3):
                    u = sum(O[_plus(_unit(i), _plus(_unit(j), _unit(k)))] * r[j] * r[k]
                            for j in range(3) for k in range(3))
                    tr = sum(O[_plus(_unit(i), tuple(2 * v for v in _unit(j)))] for j in range(3))
                    F.append(7.5 * u * R2 ** -3.5 - 1.5 * tr * R2 ** -2.5)
            else:
                F = [-sum((-1) ** sum(q) / (_factorial(p) * _factorial(q)) * tgt[p] * src[q] * D[_plus(_plus(p, q), _unit(k))]
                          for p, q in itertools.product(src, src) if sum(p) + sum(q) == P) for k in range(3)]
            for k in range(3):
                L[_unit(k)].index_add_(0, T, -F[k] / tgt[(0, 0, 0)])
    return L


def _near_field(t, near, eps2):
    acc = [torch.zeros_like(t.m) for _ in range(3)]
    A, B = near
    size = t.count[A] * t.count[B]
    ends = torch.cumsum(size, 0)
    total, at, done = int(ends[-1]), 0, 0
    while done < total:
        to = max(at + 1, int(torch.searchsorted(ends, done + (1 << 24), right=True)))
        a, b, k = A[at:to], B[at:to], size[at:to]
        row = torch.repeat_interleave(torch.arange(a.shape[0], device=k.device), k)
        j = torch.arange(row.shape[0], device=k.device) - (torch.cumsum(k, 0) - k)[row]
        nb = t.count[b][row]
        i, j = t.begin[a][row] + j // nb, t.begin[b][row] + j % nb
        d = [v[j] - v[i] for v in t.x]
        r2 = (d[0] ** 2 + d[1] ** 2) + d[2] ** 2
        w = torch.where(r2 > 0, (r2 + eps2).pow(-1.5), torch.zeros_like(r2))
        other = (a != b)[row]
        for c in range(3):
            acc[c].index_add_(0, i, t.m[j] * d[c] * w)
            acc[c].index_add_(0, j, torch.where(other, -t.m[i] * d[c] * w, torch.zeros_like(w)))
        done, at = int(ends[to - 1]), to
    return acc


def _accelerations(x, m, case):
    P, eps2 = case["order"], case["eps"] ** 2
    t = _Tree(x, m, case["n_crit"], P)
    far, near = _walk(t, case["theta"])
    L = _far_field(t, far, case["variant"], P, eps2)
    acc = _near_field(t, near, eps2)
    for lo, hi in t.levels:  # down the tree: shift to the children, evaluate at the bodies of the leaves
        cells = torch.arange(lo, hi, device=m.device)
        par = cells[~t.leaf[cells]]
        k = t.nchild[par]
        if par.shape[0]:
            own = torch.repeat_interleave(par, k)
            kid = torch.repeat_interleave(t.first[par] - (torch.cumsum(k, 0) - k), k) + torch.arange(
                own.shape[0], device=m.device)
            w = _powers([z[kid] - z[own] for z in t.Z], P - 1)
            up = {a: v[own] for a, v in L.items()}
            for a in L:
                L[a][kid] += sum(up[_plus(a, b)] * w[b] / _factorial(b) for b in w if sum(a) + sum(b) <= P)
        cell, at = t.bodies(cells[t.leaf[cells]])
        w = _powers([v[at] - z[cell] for v, z in zip(t.x, t.Z)], P - 1)
        for c in range(3):
            acc[c][at] -= sum(L[_plus(a, _unit(c))][cell] * w[a] / _factorial(a) for a in w)
    out = [torch.empty_like(v) for v in acc]
    for c in range(3):
        out[c][t.order] = acc[c]
    return out


def exact(case, seed):
    if case["kind"] == "selector":  # which pairs interact is the network's decision, in BF16
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    up = lambda *v: [torch.from_numpy(a).to(dev) for a in v]  # noqa: E731
    if case["kind"] == "forest":
        off, b = _forest(case, seed)
        x, m = up(b.x, b.y, b.z), up(b.m)[0]
        parts = [_accelerations([v[s:e] for v in x], m[s:e], case) for s, e in zip(off[:-1], off[1:])]
        return [torch.cat([p[c] for p in parts]) for c in range(3)]
    b = _system(case, seed)
    x, m = up(b.x, b.y, b.z), up(b.m)[0]
    a = _accelerations(x, m, case)
    if case["kind"] != "leapfrog":
        return a
    v, dt, mom = up(b.vx, b.vy, b.vz), _timestep(), []

    def totals():
        cross = [x[1] * v[2] - x[2] * v[1], x[2] * v[0] - x[0] * v[2], x[0] * v[1] - x[1] * v[0]]
        mom.append(torch.stack([(m * q).sum() for q in v + cross]))

    totals()
    for _ in range(LEAP_STEPS):
        v = [p + q * (0.5 * dt) for p, q in zip(v, a)]
        x = [p + q * dt for p, q in zip(x, v)]
        a = _accelerations(x, m, case)
        v = [p + q * (0.5 * dt) for p, q in zip(v, a)]
        totals()
    return {"state": x + v, "acc": a, "mom": torch.stack(mom)}
