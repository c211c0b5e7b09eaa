"""Interaction lists of the walk by records of eight pairs: generations of one
record up to several rounds per tile, cells with one to eight children (pairs of
a cell's children with themselves take up to five records), against the oracle's
lists; and the order of the lists, which must not depend on the run."""
import numpy as np
import pytest

import oracle
from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _lists(p, m, theta, n_crit, s=None):
    from paper_1706_06989_gb300 import fmm
    s = s or fmm.FMM(theta=theta, n_crit=n_crit)
    s.solve(*(torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m)))
    return s, [v.cpu().numpy() for v in s.export_lists()]


def _canon(p):
    p = np.sort(np.asarray(p, dtype=np.int64).reshape(-1, 2), axis=1)
    return np.sort(p[:, 0] << 32 | p[:, 1])


@pytest.mark.parametrize("n,theta,n_crit", [(2, 0.5, 1), (9, 0.5, 1), (70, 0.5, 1), (700, 0.8, 1), (6000, 0.5, 1),
                                            (20000, 0.3, 4), (60000, 0.5, 2)])
@pytest.mark.parametrize("kind", ["cube", "plummer", "line"])
def test_lists_match_oracle(kind, n, theta, n_crit):
    p = (ics.uniform_cube(n, seed=n) if kind == "cube" else ics.plummer(n, seed=n)).pos()
    if kind == "line":  # cells of one or two children
        p = p[:, :1] * np.array([[1.0, 1.0, 1.0]]) + 1e-9 * p
    m = np.full(n, 1.0 / n)
    s, got = _lists(p, m, theta, n_crit)
    o = oracle.Oracle(p[:, 0].copy(), p[:, 1].copy(), p[:, 2].copy(), m, theta, n_crit)
    want = o.lists()
    assert np.array_equal(_canon(got[0]), _canon(want[0]))
    assert np.array_equal(_canon(got[1]), _canon(want[1]))
    assert np.array_equal(np.sort(got[2]), np.sort(want[2]))
    _, again = _lists(p, m, theta, n_crit, s)
    assert all(np.array_equal(a, b) for a, b in zip(got, again))
