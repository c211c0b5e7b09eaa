"""The softened FP64 near field: a pair far closer than the softening length, where
the window rounds positions (close to the coordinate planes), is good to its own
magnitude.  On the host (the kernel's steps on its arithmetic) and on the GPU."""
import numpy as np
import pytest

import near_field_model
import oracle


@pytest.fixture(scope="module")
def near_sum(tmp_path_factory):
    return near_field_model.build(str(tmp_path_factory.mktemp("soft")))


def _group(d, heavy, seed=0, n=30):
    """n bodies of mass 1 in the unit cube and two of mass `heavy` within d of its
    centre, which is the coordinate origin."""
    rng = np.random.default_rng(seed)
    p = np.vstack([rng.normal(size=(2, 3)) * d, rng.uniform(-0.5, 0.5, (n, 3))])
    return p, np.r_[heavy, heavy, np.ones(n)]


LENGTHS = [2.0 ** -9, 2.0 ** -8, 2.0 ** -7, 2.0 ** -6, 2.0 ** -5, 2.0 ** -4, 0.2, 1.0, 3.0, 100.0, 1e8]


@pytest.mark.parametrize("eps", LENGTHS)
@pytest.mark.parametrize("d", [1e-2, 1e-4, 1e-5, 1e-6, 1e-8, 1e-10])
@pytest.mark.parametrize("heavy", [1.0, 10.0, 1000.0])
def test_terms_are_good_to_their_own_magnitude(near_sum, eps, d, heavy):
    """A difference is good to 2^-57 of the window and at least 2^-7 of it (else the
    pair is evaluated in FP64, to 2^-50), the factor to 2^-54: 2^-49 of a term."""
    for seed in range(10):
        p, m = _group(d, heavy, seed)
        for i in (0, 1, 2):
            s, ms = np.delete(p, i, 0), np.delete(m, i)
            got, _ = near_sum(p[i], s, ms, eps=eps)
            ref, size = near_field_model.exact(p[i], s, ms, eps)
            assert np.sqrt(((got - ref) ** 2).sum()) <= 2.0 ** -49 * size, (seed, i)


@pytest.mark.gpu
@pytest.mark.parametrize("eps", LENGTHS)
@pytest.mark.parametrize("d", [1e-2, 1e-4, 1e-5, 1e-6, 1e-8, 1e-10])
def test_gpu_matches_exact_sums(eps, d):
    """One leaf: direct sums only.  2^-49 of every term, and as much for what the
    sums over 32 terms and the reference round."""
    torch = pytest.importorskip("torch")
    from paper_1706_06989_gb300 import fmm
    for heavy in (1.0, 10.0, 1000.0):
        p, m = _group(d, heavy)
        x, y, z = (np.ascontiguousarray(p[:, k]) for k in range(3))
        s = fmm.FMM(theta=0.3, n_crit=len(m))
        s.set_softening(eps)
        got = torch.stack(s.solve(*(torch.from_numpy(v).cuda() for v in (x, y, z, m))), 1).cpu().numpy()
        ref = oracle.direct(x, y, z, m, eps=eps)
        size = np.array([near_field_model.exact(p[i], p, m, eps)[1] for i in range(len(m))])
        assert (np.linalg.norm(got - ref, axis=1) <= 2.0 ** -48 * size).all()
