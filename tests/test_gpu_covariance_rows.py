"""rpba_covariance for more ids than the staging array holds at a time: every row
is that of its own id, whatever its place in the call (the same arithmetic per
point: equal bits)."""

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_rows_do_not_depend_on_their_place(precision):
    prob = synth.config(1)
    g = rpba.Rpba(prob, precision=precision)
    g.intersect()
    one = np.concatenate([g.covariance([j]) for j in range(40)])
    rng = np.random.default_rng(2)
    # one staging array holds at least 3 N doubles and a row takes 9.5
    for n in (2, 3 * g.N // 9, 3 * g.N // 9 + 1, 5 * g.N + 1):
        ids = rng.integers(0, 40, n)
        np.testing.assert_array_equal(g.covariance(ids), one[ids])
    with pytest.raises(rpba.RpbaError):
        g.covariance(np.r_[np.zeros(5 * g.N, int), g.N])


def test_smallest_block():
    prob = synth.config(1)
    keep = np.flatnonzero(prob["obs_point"] == prob["obs_point"][0])
    assert keep.size >= 2
    small = dict(prob, points=prob["points"][prob["obs_point"][0]][None], obs_cam=prob["obs_cam"][keep],
                 obs_point=np.zeros(keep.size, np.int32), obs_xy=prob["obs_xy"][keep])
    if prob.get("obs_winv") is not None:
        small["obs_winv"] = prob["obs_winv"][keep]
    g = rpba.Rpba(small)
    g.intersect()
    a = g.covariance([0, 0, 0])
    assert np.isfinite(a).all()
    np.testing.assert_array_equal(a[0], a[2])
