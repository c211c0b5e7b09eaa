"""The leaf tile belongs to the mixed form: in FP64 the autotuner times a leaf size once,
and a captured solve outlives fmm_set_tile."""
import numpy as np
import pytest

from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _dev(b):
    return tuple(torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (b.x, b.y, b.z, b.m))


def test_autotune_times_a_leaf_size_once():
    from paper_1706_06989_gb300 import fmm
    off, b = ics.ensemble(nsys=8, seed=6, nmin=500, nmax=3000)
    s = fmm.FMM(theta=0.5)
    _, tile, table = s.autotune(*_dev(b), off, ncrit=(16, 32), tiles=(32, 8, 16), reps=2)
    assert tile == 32
    for n in (16, 32):
        assert len({table[(n, t)] for t in (8, 16, 32)}) == 1 and table[(n, 8)] > 0


@pytest.mark.parametrize("precision,captures", [("fp64", 1), ("mixed", 2)])
def test_graph_and_tile(precision, captures):
    from paper_1706_06989_gb300 import fmm
    x, y, z, m = _dev(ics.plummer(5000, seed=2))
    s = fmm.FMM(theta=0.5, precision=precision)
    s.set_graph(True)
    out = tuple(torch.empty_like(x) for _ in range(3))
    s.solve(x, y, z, m, out)
    first = torch.stack(out)
    s.set_tile(32)
    s.solve(x, y, z, m, out)
    gs = s.graph_stats()
    assert gs["captures"] == captures and gs["replays"] == 2 - captures
    if precision == "fp64":
        assert torch.equal(torch.stack(out), first)
