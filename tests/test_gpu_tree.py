"""The octree built from all levels at once against the oracle's: leaf sizes at
the edges of a block's windows, chains of single-child cells, coincident
bodies, forests."""
import numpy as np
import pytest

import oracle
from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FIELDS = ("begin", "count", "level", "parent", "first_child", "nchild")


def _bodies(kind, n):
    rng = np.random.default_rng(n)
    p = ics.plummer(n, seed=3).pos()
    if kind == "chains":  # tight clumps far apart: long single-child chains
        p = np.repeat(rng.uniform(-1, 1, (n // 8, 3)), 8, axis=0)[:n]
        p = np.concatenate([p, rng.uniform(-1, 1, (n - len(p), 3))])
        p += 1e-6 * rng.normal(size=p.shape)
    elif kind == "coincident":
        p[: n // 2] = p[0]
    return np.ascontiguousarray(p), np.full(n, 1.0 / n)


def _tree(p, m, n_crit):
    from paper_1706_06989_gb300 import fmm
    x, y, z, mm = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m))
    s = fmm.FMM(n_crit=n_crit)
    s.build_tree(x, y, z, mm)
    return {k: v.cpu().numpy() for k, v in s.export_tree(geometry=False).items() if k in FIELDS}


@pytest.mark.parametrize("n_crit", [1, 25, 255, 256, 2048, 2049, 4999, 5000])
@pytest.mark.parametrize("kind", ["plummer", "chains", "coincident"])
def test_tree_matches_oracle(kind, n_crit):
    p, m = _bodies(kind, 5000)
    got = _tree(p, m, n_crit)
    c = oracle.Oracle(p[:, 0].copy(), p[:, 1].copy(), p[:, 2].copy(), m, 0.5, n_crit).cells()
    for k in FIELDS:
        assert np.array_equal(got[k], np.asarray(getattr(c, k))), k


@pytest.mark.parametrize("n_crit", [25, 300, 2500])
def test_forest_cells_are_those_of_its_systems(n_crit):
    """Leaves of a forest: the same bodies per leaf as one tree per system."""
    from paper_1706_06989_gb300 import fmm
    sizes = [1, 2, 3000, 26, 257, 700]
    parts = [_bodies("plummer", n) if n > 2 else (np.zeros((n, 3)) + np.arange(n)[:, None], np.ones(n)) for n in sizes]
    p, m = np.concatenate([q[0] for q in parts]), np.concatenate([q[1] for q in parts])
    off = np.concatenate([[0], np.cumsum(sizes)])
    x, y, z, mm = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m))
    s = fmm.FMM(n_crit=n_crit)
    s.solve_batch(x, y, z, mm, off)
    t = {k: v.cpu().numpy() for k, v in s.export_tree(geometry=False).items() if k in FIELDS}
    leaf = t["nchild"] == 0
    got = {(int(b), int(c)) for b, c in zip(t["begin"][leaf], t["count"][leaf])}
    want = set()
    for (q, mass), o in zip(parts, off):
        u = _tree(q, mass, n_crit)
        lf = u["nchild"] == 0
        want |= {(int(b + o), int(c)) for b, c in zip(u["begin"][lf], u["count"][lf])}
    assert got == want
