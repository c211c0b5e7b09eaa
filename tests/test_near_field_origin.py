"""The FP64 near field next to the coordinate planes, where windows and the 96-bit
positions round: on the host, no less accurate than FP64 arithmetic."""
import numpy as np
import pytest

import near_field_model


@pytest.fixture(scope="module")
def near_sum(tmp_path_factory):
    return near_field_model.build(str(tmp_path_factory.mktemp("origin")))


def _fp64(t, s, m):
    d = t - s
    r2 = (d * d).sum(1)
    ri = 1.0 / np.sqrt(r2)
    return ((m * (ri * ri * ri))[:, None] * d).sum(0)


def _rms(near_sum, log2_r, masses, size=1.0):
    """rms errors, against the sum of the terms, of a pair about the origin at
    2^log2_r of the window that a far body sets: (fixed point, FP64 arithmetic).
    Pairs that the fixed point leaves to FP64 are FP64 arithmetic themselves."""
    rng = np.random.default_rng(1)
    errors = []
    for _ in range(1000):
        u = rng.normal(size=3)
        u *= 2.0 ** (log2_r + 1) / np.linalg.norm(u)
        a = rng.normal(size=3) * 2.0 ** (log2_r - 1)
        s, t = size * np.vstack([a, np.full(3, rng.uniform(0.55, 0.99))]), size * (a + u)
        got, how = near_sum(t, s, masses, err=float(rng.uniform(-2.4e-7, 2.4e-7)), extent=1.0)
        if how[0] == 2:
            continue
        ref, total = near_field_model.exact(t, s, masses)
        errors.append([np.sqrt(float(((v - ref) ** 2).sum())) / total for v in (got, _fp64(t, s, masses))])
    return np.sqrt((np.array(errors) ** 2).mean(0)) if errors else (0.0, 0.0)


@pytest.mark.parametrize("log2_r", [-12, -10, -8, -7.5, -7, -6.5, -6, -5.5, -5, -4, -3])
def test_pairs_in_rounded_windows(near_sum, log2_r):
    fixed, fp64 = _rms(near_sum, log2_r, np.array([1.0, 1e-3]))
    assert fixed <= fp64


@pytest.mark.parametrize("log2_r", [-16, -14, -12])
@pytest.mark.parametrize("log2_size", [-29, -28, -26, -20])
def test_pairs_close_to_the_resolution_of_positions(near_sum, log2_r, log2_size):
    """A light pair beside a body that is heavier by 2^20, all in a small part of the
    system about the origin: still 2^-42 of the system apart and further, or in FP64."""
    fixed, fp64 = _rms(near_sum, log2_r, np.array([2.0 ** -20, 1.0]), 2.0 ** log2_size)
    assert fixed <= fp64
