"""Moments of the general orders against their definition, in long double, at
leaves below and above a warp's 32 bodies, and the trace relation of the locals
that the M2L's reduced sums leave to be restored."""
import numpy as np
import pytest

from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _multi(P):
    return [(a, b, n - a - b) for n in range(P + 1) for a in range(n, -1, -1) for b in range(n - a, -1, -1)]


def _solve(P, n, n_crit):
    from paper_1706_06989_gb300 import fmm
    p = ics.plummer(n, seed=n_crit).pos()
    m = np.random.default_rng(P).uniform(0.1, 1.0, n)
    s = fmm.FMM(theta=0.7, n_crit=n_crit, order_P=P)
    s.solve(*(torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m)))
    return s, p, m


@pytest.mark.parametrize("P", [4, 5, 6, 7, 8])
@pytest.mark.parametrize("n,n_crit", [(2, 1), (200, 1), (900, 33), (900, 100), (64, 64)])
def test_moments_match_definition(P, n, n_crit):
    s, p, m = _solve(P, n, n_crit)
    t = {k: v.cpu().numpy() for k, v in s.export_tree().items()}
    order = s.export_keys()[1].cpu().numpy()
    got = s.export_moments().cpu().numpy()
    mi = np.array(_multi(P))
    X, mu = p[order].astype(np.longdouble), m[order].astype(np.longdouble)
    # a leaf's sum: n_crit terms of up to P + 1 roundings each; a level's shift:
    # three sums of up to P + 1 terms, scaled twice, and a sum of eight; terms of
    # order k are at most M (3 R)^k, shifts being within R and child radii 2 R
    depth = int(t["level"].max())
    eps = 2.0**-52 * (n_crit + P + 8 + depth * (3 * (P + 1) + 18))
    for c in range(len(t["begin"])):
        b, e = t["begin"][c], t["begin"][c] + t["count"][c]
        d = X[b:e] - t["Z"][c]
        want = np.array([(mu[b:e] * d[:, 0]**i * d[:, 1]**j * d[:, 2]**k).sum() for i, j, k in mi])
        assert (np.abs(got[c] - want) <= eps * t["M"][c] * (3 * t["Rmax"][c]) ** mi.sum(1)).all(), c


@pytest.mark.parametrize("P", [4, 5, 6, 7, 8])
def test_locals_are_harmonic(P):
    s, _, _ = _solve(P, 900, 33)
    loc = s.export_locals().cpu().numpy()
    idx = {a: i - 1 for i, a in enumerate(_multi(P))}
    for i, j, k in _multi(P - 2):
        parts = loc[:, [idx[(i + 2, j, k)], idx[(i, j + 2, k)], idx[(i, j, k + 2)]]]
        # restored from at most 2^4 reduced coefficients and shifted down at most
        # 8 levels with 3 (P + 1) + 16 roundings each: 8 * 43 * 16 * 2^-52 = 1.2e-12
        same = np.array([idx[a] for a in _multi(P) if sum(a) >= i + j + k + 2])
        scale = np.abs(loc[:, same]).max(1)
        assert (np.abs(parts.sum(1)) <= 1e-11 * scale).all()
