"""Which pairs the FP64 near field's integers take: all but those closer than 2^-6 of
their batch's window (on the host; the FP64 path that takes the others gives right
sums too, so that no test of results sees a wrong limit)."""
import numpy as np
import pytest

import near_field_model


@pytest.fixture(scope="module")
def near_sum(tmp_path_factory):
    return near_field_model.build(str(tmp_path_factory.mktemp("taken")))


@pytest.mark.parametrize("kind", ["plain", "offset", "origin", "grid", "close", "masses"])
@pytest.mark.parametrize("log2_unit", [-90, 0, 90])
def test_only_close_pairs_are_left(near_sum, kind, log2_unit):
    """The heaviest source of a class gets k >= 18 at the window's bound and loses
    three per octave, so it fits down to 2^-6; light ones further.  The window is at
    most twice the largest offsets from the first source, of the target and of a
    source, together (and 2^-26 of the extent, which they are rounded up by).  A pair
    takes a window of its own from 2^-5 on at the earliest."""
    rng = np.random.default_rng(11)
    taken = 0
    for trial in range(100):
        ns = int(rng.integers(1, 130))
        size = 10.0 ** rng.uniform(-3, 0)
        centre = {"origin": 0.0, "offset": 1e3}.get(kind, 1.0) * rng.uniform(-1, 1, 3)
        t = centre + size * rng.uniform(-1, 1, 3)
        s = centre + size * rng.uniform(-1, 1, (ns, 3))
        m = rng.uniform(0.1, 1.0, ns)
        if kind == "close":
            s[::3] = t + size * 10.0 ** rng.uniform(-12, -1, (len(s[::3]), 1)) * rng.normal(size=(len(s[::3]), 3))
        if kind == "masses":
            m = 10.0 ** rng.uniform(-12, 12, ns)
        if kind == "grid":
            t, s = np.round(t * 64) / 64, np.round(s * 64) / 64
        _, how = near_sum(t * 2.0 ** log2_unit, s * 2.0 ** log2_unit, m, extent=4.0 * 2.0 ** log2_unit)
        for j0 in range(0, ns, 32):
            b, h = s[j0:j0 + 32], how[j0:j0 + 32]
            window = 2 * (np.abs(t - s[0]).max() + np.abs(b - s[0]).max() + 4 * 2.0 ** -26)
            r = np.linalg.norm(b - t, axis=1)
            assert (h[r > 2.0 ** -6 * window] != 2).all() and (h[r > 2.0 ** -5 * window] == 0).all(), trial
        taken += int((how == 0).sum())
    assert taken > 100 * 30
