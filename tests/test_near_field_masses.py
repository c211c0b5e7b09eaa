"""The FP64 near field's sums where masses differ widely: light bodies close together
with a heavy one far away, or in their midst.  On the host (the kernel's steps on its
arithmetic) and on the GPU."""
import numpy as np
import pytest

import near_field_model
import oracle


@pytest.fixture(scope="module")
def near_sum(tmp_path_factory):
    return near_field_model.build(str(tmp_path_factory.mktemp("masses")))


def _system(size, log2_light, heavies, seed=0, n=40):
    """n light bodies in a cube of the given size and `heavies` of mass 1 around
    it, 0.2 to 0.6 away (-1: one heavy body in the cube)."""
    rng = np.random.default_rng(seed)
    c = np.array([0.3, 0.21, 0.13])
    p, m = c + size * rng.uniform(-0.5, 0.5, (n, 3)), 2.0 ** log2_light * rng.uniform(0.5, 1.0, n)
    if heavies < 0:
        m[5] = 1.0
        q = c + rng.uniform(0.2, 0.6, (3, 3))
        return np.vstack([p, q]), np.r_[m, np.full(3, m[0])]
    return np.vstack([p, c + rng.uniform(0.2, 0.6, (heavies, 3))]), np.r_[m, rng.uniform(0.5, 1.0, heavies)]


SIZES, LIGHT, HEAVIES = [0.5, 1e-1, 1e-2, 1e-3, 1e-4, 1e-6], [0, -7, -10, -20, -27, -33, -40, -60], [-1, 1, 8, 40]


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("log2_light", LIGHT)
@pytest.mark.parametrize("heavies", HEAVIES)
def test_sums_are_good_to_their_terms(near_sum, size, log2_light, heavies):
    """Every term is within 2^-49 of the sum of the terms' magnitudes (its
    difference, its factor and the sums' unit), and only pairs closer than 2^-6 of
    their batch's window are left to FP64: it is at most twice the largest offsets
    from the first source, of the target and of a source, together (and 2^-26 of the
    extent, which they are rounded up by)."""
    p, m = _system(size, log2_light, heavies)
    for i in (0, 5, 7, len(m) - 1):
        for own in (False, True):
            s, ms = (p, m) if own else (np.delete(p, i, 0), np.delete(m, i))
            got, how = near_sum(p[i], s, ms, own=i if own else -1, extent=2.0)
            ref, total = near_field_model.exact(p[i], s, ms)
            assert np.sqrt(((got - ref) ** 2).sum()) <= 2.0 ** -49 * total, (i, own)
            for j0 in range(0, len(s), 32):
                b = s[j0:j0 + 32]
                window = 2 * (np.abs(p[i] - s[0]).max() + np.abs(b - s[0]).max() + 2.0 ** -26)
                left = np.linalg.norm(b - p[i], axis=1)[how[j0:j0 + 32] == 2]
                assert (left <= 2.0 ** -6 * window).all(), (i, own)


@pytest.mark.gpu
@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("log2_light", LIGHT)
def test_gpu_matches_exact_sums(size, log2_light):
    """theta so small that no pair of cells with a radius is accepted.  2^-49 of every term,
    and as much for what the sums of the parts and the reference round."""
    torch = pytest.importorskip("torch")
    from paper_1706_06989_gb300 import fmm
    for heavies in HEAVIES:
        for n_crit in (10, 100):
            p, m = _system(size, log2_light, heavies)
            x, y, z = (np.ascontiguousarray(p[:, k]) for k in range(3))
            s = fmm.FMM(theta=1e-9, n_crit=n_crit)
            got = torch.stack(s.solve(*(torch.from_numpy(v).cuda() for v in (x, y, z, m))), 1).cpu().numpy()
            ref = oracle.direct(x, y, z, m)
            bound = 2.0 ** -48 * np.array([near_field_model.exact(p[i], p, m)[1] for i in range(len(m))])
            if s.stats().n_m2l:
                # cells of one body have no radius and are accepted at any angle:
                # their centres, quotients of rounded sums, are good to a few units
                # in the last place of the coordinates
                d = np.linalg.norm(p[None] - p[:, None], axis=2)
                bound += 16 * 2.0 ** -53 * np.abs(p).max() * (m[None] / np.where(d > 0, d, np.inf) ** 3).sum(1)
            assert (np.linalg.norm(got - ref, axis=1) <= bound).all(), (heavies, n_crit)
