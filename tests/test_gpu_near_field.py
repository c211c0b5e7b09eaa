"""The FP64 near field in fixed point against exact direct sums: leaf sizes at the
edges of the row blocks and entry groups, close and coincident bodies, wide
mass ranges, systems off the origin, softening lengths inside and beyond the
window."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _system(kind, n):
    rng = np.random.default_rng(n + sum(map(ord, kind)))
    p = rng.uniform(-0.5, 0.5, (n, 3))
    m = rng.uniform(0.5, 1.0, n)
    if kind == "offset":
        p = p + np.array([1e5, -3e4, 7.0])
    elif kind == "close":  # companions from 1e-13 to 1e-2 of the system, two of them coincident
        k = n // 2
        p[k:2 * k] = p[:k] + 10.0 ** rng.uniform(-13, -2, (k, 1)) * rng.normal(size=(k, 3))
        p[1] = p[0]
    elif kind == "masses":
        m = 2.0 ** rng.uniform(-45, 45, n)
    elif kind == "cluster":  # a dense core beside sparse bodies
        p[: n // 2] *= 1e-5
    elif kind == "tiny":
        p *= 2.0 ** -90
    return p, m


def _sizes(p, m, eps=0.0):
    """Sum of the magnitudes of every body's pair terms."""
    d = p[None] - p[:, None]
    r2 = np.sum(d * d, axis=2)
    r = np.sqrt(r2)
    t = m[None] * r / np.where(r2 > 0, r2 + eps * eps, 1.0) ** 1.5
    return np.where(r2 > 0, t, 0.0).sum(1)


@pytest.mark.parametrize("n_crit", [1, 7, 16, 17, 33, 400])
@pytest.mark.parametrize("kind", ["cube", "offset", "close", "masses", "cluster", "tiny"])
def test_near_field_matches_direct_sums(kind, n_crit):
    """theta so small that no pair of cells is accepted: direct sums only."""
    from paper_1706_06989_gb300 import fmm
    p, m = _system(kind, 400)
    x, y, z, mm = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m))
    s = fmm.FMM(theta=1e-7, n_crit=n_crit)
    got = torch.stack(s.solve(x, y, z, mm), 1).cpu().numpy()
    st = s.stats()
    ref = oracle.direct(p[:, 0].copy(), p[:, 1].copy(), p[:, 2].copy(), m)
    bound = 1e-14 * _sizes(p, m)
    if st.n_m2l:
        # cells of one body (or of coincident bodies) have no radius and are
        # accepted at any angle: their centres, quotients S / M of rounded
        # sums, are good to a few units in the last place of the coordinates
        d = np.linalg.norm(p[None] - p[:, None], axis=2)
        bound += 16 * 2.0 ** -53 * np.abs(p).max() * (m[None] / np.where(d > 0, d, np.inf) ** 3).sum(1)
    assert (np.linalg.norm(got - ref, axis=1) <= bound).all()
    assert st.p2p_body_pairs <= 400 * 399 // 2 and (st.n_m2l or st.p2p_body_pairs == 400 * 399 // 2)


@pytest.mark.parametrize("eps", [1e-9, 1e-3, 0.2, 3.0, 1e6])
@pytest.mark.parametrize("kind", ["cube", "close"])
def test_softened_near_field_matches_oracle(kind, eps):
    from paper_1706_06989_gb300 import fmm
    p, m = _system(kind, 300)
    x, y, z, mm = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m))
    s = fmm.FMM(theta=0.3, n_crit=300)  # one leaf: direct sums only
    s.set_softening(eps)
    got = torch.stack(s.solve(x, y, z, mm), 1).cpu().numpy()
    ref = oracle.direct(p[:, 0].copy(), p[:, 1].copy(), p[:, 2].copy(), m, eps=eps)
    # against the size of the summed terms: far beyond the separations the
    # softened forces nearly cancel
    assert (np.linalg.norm(got - ref, axis=1) / _sizes(p, m, eps)).max() <= 1e-14
