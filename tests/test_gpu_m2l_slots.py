"""The FP64 cell interactions and their per-cell sums where cells have few
partners (none, one, an odd number, just above a step of the sums): systems of
one body per leaf, unsoftened and softened, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [2, 3, 4, 5, 8, 9, 10, 17, 33, 100])
@pytest.mark.parametrize("variant", ["UC", "TC", "TCO"])
@pytest.mark.parametrize("eps", [0.0, 1e-3])
def test_few_partners(n, variant, eps):
    from paper_1706_06989_gb300 import fmm
    p = ics.plummer(n, seed=5).pos()
    m = np.random.default_rng(n).uniform(0.1, 1.0, n)
    s = fmm.FMM(theta=1.0, n_crit=1, variant=variant)
    if eps:
        s.set_softening(eps)
    a = s.solve(*(torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (p[:, 0], p[:, 1], p[:, 2], m)))
    a = torch.stack(a, 1).cpu().numpy()
    o = oracle.Oracle(p[:, 0].copy(), p[:, 1].copy(), p[:, 2].copy(), m, 1.0, 1, softening=eps)
    ref = o.accel(variant)
    assert (np.linalg.norm(a - ref, axis=1) <= 1e-12 * np.linalg.norm(ref, axis=1)).all()
