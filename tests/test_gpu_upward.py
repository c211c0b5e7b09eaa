"""Upward pass on both sides of each split of its work (leaves per warp, parents
per warp) and R_max through its FP32 filter, also far from the origin and at
extreme units: M, Z, R_max to the bit, moments within their rounding."""
import numpy as np
import pytest

import oracle
from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ORDER = np.repeat([0, 1, 2, 3], [1, 3, 6, 10])


def _check(p, m, n_crit, moments=True):
    from paper_1706_06989_gb300 import fmm
    p = np.ascontiguousarray(p)
    x, y, z, mm = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m))
    s = fmm.FMM(n_crit=n_crit)
    s.solve(x, y, z, mm)
    t = s.export_tree()
    o = oracle.Oracle(p[:, 0].copy(), p[:, 1].copy(), p[:, 2].copy(), m, 0.5, n_crit)
    M, Z, R, want = (np.asarray(v) for v in o.geometry())
    for key, ref in (("M", M), ("Z", Z), ("Rmax", R)):
        assert np.array_equal(t[key].cpu().numpy().view(np.int64), ref.view(np.int64)), key
    if not moments:
        return
    got = s.export_moments().cpu().numpy()[:, :20]
    # a moment is a sum of at most n_crit (leaf) or eight (parent, per level)
    # terms with about eight roundings each; the terms of order k are at most
    # M (3 R)^k, since shifts are within R and child radii within 2 R
    depth = int(t["level"].max()) + 1
    tol = 2 * (n_crit + 16 * depth) * 2.0**-52 * M[:, None] * (3 * R[:, None]) ** ORDER
    keep = ORDER != 1  # dipoles are zero up to the rounding of Z itself
    assert (np.abs(got - want[:, :20]) <= tol)[:, keep].all()


@pytest.mark.parametrize("n,n_crit", [(1, 1), (2, 1), (33, 40), (700, 33), (2300, 1), (2700, 1), (5200, 1), (11000, 1),
                                      (40000, 2), (30000, 200)])
def test_upward_matches_oracle(n, n_crit):
    b = ics.plummer(max(n, 2), seed=n).pos()[:n]
    m = np.random.default_rng(n).uniform(0.1, 1.0, n)
    _check(b, m, n_crit)


@pytest.mark.parametrize("scale,shift", [(1.0, 1e7), (1e-18, 0.0), (1e-16, 1e-3), (1e17, 1e19), (1e22, 0.0)])
@pytest.mark.parametrize("n_crit", [8, 64])
def test_rmax_filter_units(scale, shift, n_crit):
    b = ics.plummer(4000, seed=9).pos() * scale + shift
    # far from the origin the child dipoles, which the shift leaves out, carry
    # the rounding of the coordinates: the moments have no bound of their own
    _check(b, np.full(4000, 1.0 / 4000), n_crit, moments=False)
