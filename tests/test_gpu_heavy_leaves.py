"""Mixed near field of leaves with many columns, whose rows and columns become
items of their own: leaves of one body, of a few, of more than two row groups,
column counts around an item's 512 and a chunk's 4096; against the oracle with
the mixed form's accuracy, and reproducible to the bit."""
import numpy as np
import pytest

import oracle
from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,n_crit", [(512, 1), (515, 2), (1100, 3), (1500, 5), (5000, 40), (9000, 70)])
@pytest.mark.parametrize("tile", [8, 16, 32])
@pytest.mark.parametrize("eps", [0.0, 0.05])
def test_all_pairs_direct(n, n_crit, tile, eps):
    from paper_1706_06989_gb300 import fmm
    p = ics.uniform_cube(n, seed=n).pos()
    m = np.random.default_rng(n).uniform(0.5, 1.0, n) / n
    d = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m)]
    s = fmm.FMM(theta=1e-4, n_crit=n_crit, precision="mixed")  # no cell pair of several bodies is accepted
    s.set_tile(tile)
    if eps:
        s.set_softening(eps)
    a = torch.stack(s.solve(*d), 1).cpu().numpy()
    o = oracle.Oracle(p[:, 0].copy(), p[:, 1].copy(), p[:, 2].copy(), m, 1e-4, n_crit, softening=eps)
    ref = o.accel("TC")
    dev = np.linalg.norm(a - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.sqrt(np.mean(dev**2)) <= 1e-6
    b = torch.stack(s.solve(*d), 1).cpu().numpy()
    assert np.array_equal(a, b)


def test_outlying_leaves():
    """A dense cluster and a few far bodies: their leaves meet every other one."""
    from paper_1706_06989_gb300 import fmm
    p = ics.plummer(30000, seed=3).pos()
    p[:40] *= 300.0
    m = np.full(len(p), 1.0 / len(p))
    d = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m)]
    s = fmm.FMM(theta=0.4, n_crit=25, precision="mixed")
    a = torch.stack(s.solve(*d), 1).cpu().numpy()
    ref = oracle.Oracle(p[:, 0].copy(), p[:, 1].copy(), p[:, 2].copy(), m, 0.4, 25).accel("TC")
    dev = np.linalg.norm(a - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.sqrt(np.mean(dev**2)) <= 1e-6


def test_partials_at_the_ends_of_the_float_range():
    """Partners' partials of any size are widened exactly: masses from 1e-30 to
    1e30 in one system, every pair summed directly."""
    from paper_1706_06989_gb300 import fmm
    p = ics.uniform_cube(600, seed=4).pos()
    m = 10.0 ** np.random.default_rng(4).uniform(-30, 30, 600)
    d = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m)]
    a = torch.stack(fmm.FMM(theta=1e-4, n_crit=4, precision="mixed").solve(*d), 1).cpu().numpy()
    ref = oracle.direct(p[:, 0].copy(), p[:, 1].copy(), p[:, 2].copy(), m)
    dev = np.linalg.norm(a - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert np.sqrt(np.mean(dev**2)) <= 1e-6
