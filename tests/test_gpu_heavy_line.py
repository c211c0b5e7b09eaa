"""Which leaves of the mixed near field are worked on in parts: outlying leaves whose
columns one warp would work on long after the others, but not the leaves of a solve
whose chunks are all alike."""
import pytest

from paper_1706_06989_gb300 import ics

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _near_ms(b, **kw):
    from paper_1706_06989_gb300 import fmm
    x, y, z, m = (torch.from_numpy(v).cuda() for v in (b.x, b.y, b.z, b.m))
    s = fmm.FMM(precision="mixed", **kw)
    s.set_timing(True)
    ms = []
    for _ in range(5):
        s.solve(x, y, z, m)
        torch.cuda.synchronize()
        ms.append(s.stats().ms["p2p"])
    return min(ms), s.stats().p2p_body_pairs


def test_large_leaves_cost_per_pair_what_ordinary_ones_do():
    """Parts evaluate their pairs twice.  Large leaves fill the lanes better than
    leaves of up to 25 bodies do, so a pair must not cost more (within 5%); with
    every large leaf in parts it cost 1.25 times as much."""
    ms, pairs = _near_ms(ics.plummer(1048576, seed=3), n_crit=25)
    large, many = _near_ms(ics.plummer(262144, seed=3), n_crit=1024)
    assert many > 8 * pairs
    assert large / many <= 1.05 * ms / pairs
