"""rpba_covariance at the edges of the staging array its rows go through: one
row fewer than it holds, as many, one more, and several rounds. A row is nine
doubles and the id of its point (76 bytes); the array has at least a row per
point and one more, or six doubles per instance if that is larger."""

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba, synth

pytestmark = pytest.mark.gpu


def _rows(g):
    return max(6 * g.P, (g.N + 1) * 76 // 8 + 1) * 8 // 76


@pytest.mark.parametrize("instances", [False, True])  # the array sized by points, by instances
def test_rows_at_the_edge_of_the_staging_array(instances):
    # one sub-block: an instance per point; 50: most points have several
    prob = synth.config(1)
    prob["cam_subblock"] = (np.arange(prob["cam_pose"].shape[0]) if instances else
                            np.zeros(prob["cam_pose"].shape[0])).astype(np.int32)
    g = rpba.Rpba(prob)
    g.intersect()
    rows = _rows(g)
    assert (6 * g.P * 8 // 76 == rows) == instances
    one = np.concatenate([g.covariance([j]) for j in range(60)])
    rng = np.random.default_rng(4)
    for n in (rows - 1, rows, rows + 1, 2 * rows, 2 * rows + 1):
        ids = rng.integers(0, 60, n)
        np.testing.assert_array_equal(g.covariance(ids), one[ids])
    g.close()
