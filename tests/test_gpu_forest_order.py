"""Mixed form: a system gets the same bits alone and in a forest, also where leaves
with many columns are on different sides of the line for heavy ones (it follows from
the whole call): the forest's line is above the small systems' of 512 columns, and
masses over 2^60 make every order of additions show."""
import numpy as np
import pytest

from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_crit", [25, 40])
def test_forest_and_single_solves_agree_across_the_heavy_line(n_crit):
    from paper_1706_06989_gb300 import fmm
    sizes = [4000, 12000, 30000, 60000]
    parts = [ics.plummer(n, seed=n) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    m = 2.0 ** np.random.default_rng(5).uniform(-30, 30, off[-1])
    cat = [np.concatenate([getattr(p, f) for p in parts]) for f in "xyz"] + [m]
    x, y, z, mm = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in cat)
    s = fmm.FMM(theta=0.4, n_crit=n_crit, precision="mixed")
    got = torch.stack(s.solve_batch(x, y, z, mm, off))
    for a, b in zip(off[:-1], off[1:]):
        one = torch.stack(s.solve(*(v[a:b].contiguous() for v in (x, y, z, mm))))
        assert torch.equal(one, got[:, a:b]), b - a
