"""FP64: a system's moments, locals and accelerations have the same bits alone and in a
forest, although levels of many cells (of all systems) are taken by other kernels than
levels of few: systems whose levels are below and above that line."""
import numpy as np
import pytest

from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_crit", [4, 16])
def test_moments_and_locals(n_crit):
    from paper_1706_06989_gb300 import fmm
    sizes = [300, 3000, 20000, 6000, 40000]
    parts = [ics.plummer(n, seed=n + 1) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    m = 2.0 ** np.random.default_rng(7).uniform(-10, 10, off[-1])
    cat = [np.concatenate([getattr(p, f) for p in parts]) for f in "xyz"] + [m]
    x, y, z, mm = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in cat)
    s = fmm.FMM(theta=0.6, n_crit=n_crit)
    got = torch.stack(s.solve_batch(x, y, z, mm, off))
    begin, mom, loc = s.export_tree()["begin"], s.export_moments(), s.export_locals()
    for a, b in zip(off[:-1], off[1:]):
        one = torch.stack(s.solve(*(v[a:b].contiguous() for v in (x, y, z, mm))))
        cells = (begin >= int(a)) & (begin < int(b))
        assert torch.equal(s.export_moments(), mom[cells]), b - a
        assert torch.equal(s.export_locals(), loc[cells]), b - a
        assert torch.equal(one, got[:, a:b]), b - a
