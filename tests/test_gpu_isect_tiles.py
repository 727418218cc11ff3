"""The FP64 intersection (k_isect_fused_d: every form's first intersection, and
the FP64 form's tie points) flattens the observations of a tile of points over
a CTA's threads in chunks of 128. Against the FP64 oracle from the same state,
at the edges of its tiles (16 to 128 points, by the block's size) and chunks:
one point, a tile and one more, tracks longer than a chunk, tiles of 32 and of
128 points; with observation weights, masked points and tie points only.

Both sides take the same Gauss-Newton iterates to rounding (residuals of ~1e3
px at 2^-53, so ~1e-12 px per observation, amplified by at most a few
iterations): positions to 1e-6 px in image space, the same points dropped, and
refined weights to 1e-8 relative, as in test_gpu_parity.py.
"""

import numpy as np
import pytest

import oracle
from paper_1910_08138_gb300 import rpba, synth

pytestmark = pytest.mark.gpu

BLOCKS = {  # cameras nx x ny, points, observations per point, spacing, weights
    "one": (3, 2, 1, 4, 4.0, False),
    "tile": (3, 2, 16, 4, 4.0, True),
    "tile_plus_one": (3, 2, 17, 4, 4.0, False),
    "long_tracks": (16, 16, 333, 210, 0.4, True),
    "tile_32": (6, 5, 20_003, 4, 2.0, False),
    "tile_128": (6, 5, 80_001, 3, 2.0, False),
}


@pytest.mark.parametrize("name", list(BLOCKS))
@pytest.mark.parametrize("tp_only", [False, True])
def test_fp64_intersection_matches_the_oracle(name, tp_only):
    nx, ny, n, opp, spacing, weights = BLOCKS[name]
    prob = synth.tiny(seed=5, nx=nx, ny=ny, n_points=n, opp=opp, runs=[nx * ny // 2, nx * ny - nx * ny // 2],
                      spacing=spacing, oblique_deg=20, nadir_every=3, extent=(-3.0, 3.0, -3.0, 3.0))
    rng = np.random.default_rng(1)
    if weights:
        K = prob["obs_cam"].size
        a, c = rng.uniform(0.5, 2, K), rng.uniform(0.5, 2, K)
        prob["obs_winv"] = np.stack([a, rng.uniform(-0.4, 0.4, K) * np.sqrt(a * c), c], 1)
    o = oracle.Oracle(prob)
    g = rpba.Rpba(prob, precision=0)
    w = np.where(rng.random(o.K) < 0.1, 1e-4, 1.0)
    X0, act0 = o.points()
    act0[rng.random(o.N) < 0.1 if o.N > 1 else np.zeros(o.N, bool)] = 0  # points that do not take part
    for side in (o, g):
        side.set_weights(w)
        side.set_points(X0, act0)
    o.intersect(tp_only=tp_only)
    g.intersect_points(tp_only)
    Xo, ao = o.points()
    Xg, ag = g.points()
    np.testing.assert_array_equal(ag, ao)
    ids = np.nonzero(ao)[0]
    N = np.linalg.inv(o.covariance(ids))
    d = (Xg - Xo)[ids]
    px2 = np.einsum("ni,nij,nj->n", d, N, d) / np.bincount(prob["obs_point"], minlength=o.N)[ids]
    assert px2.max() <= 1e-12
    _, Wo = o.instance_state()
    _, Wg = g.instance_state()
    ip, _ = o.instances()
    keep = ao[ip] == 1
    scale = np.abs(Wo[keep]).max(1, keepdims=True)
    assert np.all(np.abs(Wg[keep] - Wo[keep]) <= 1e-8 * scale)
    g.close()
