"""Near fields whose partial sums or work items pass 2^31 - 1 are refused before
anything is sized from their counts, and the context stays usable."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_mixed_partial_sums_beyond_32_bits():
    """64 leaves of about 47,000 bodies, every pair of leaves near: a partial sum for
    every 4,096 columns and row, 3.3e9 in all."""
    from paper_1706_06989_gb300 import fmm, ics
    b = ics.uniform_cube(3_000_000, seed=1)
    x, y, z, m = (torch.from_numpy(v).cuda() for v in (b.x, b.y, b.z, b.m))
    s = fmm.FMM(theta=0.01, n_crit=60_000, precision="mixed")
    with pytest.raises(fmm.FMMError) as e:
        s.solve(x, y, z, m)
    assert e.value.code == fmm.FMM_EUNSUPPORTED and "partial sums" in str(e.value)
    assert s.stats().nleaf == 64
    few = [v[:3000].contiguous() for v in (x, y, z, m)]
    s.set_opts(theta=0.5, n_crit=25)
    got = torch.stack(s.solve(*few))
    ref = torch.stack(fmm.FMM(theta=0.5, n_crit=25, precision="mixed").solve(*few))
    assert torch.equal(got, ref)
