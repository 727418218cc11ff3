"""The FP64 form's reduced camera system where its CTAs have edges: 1, 27, 28, 29 and
57 points in one sub-block (28 instances per CTA), tracks so long that the observations
of one CTA's instances take more than one pass of 256 threads, cameras with fewer and
more than 128 observations, inactive points, weights, 6 and 8 unknowns per camera.
Bounds of test_gpu_parity.py: to FP64 rounding, 1e-10 of the largest entry."""

import numpy as np
import pytest

from paper_1910_08138_gb300 import synth
from test_gpu_intrinsics import _sync
from test_gpu_parity import prepared, sync_state

pytestmark = pytest.mark.gpu


def _check(o, g):
    for l in range(o.L):
        So, yo = o.rcs(l, 1e-3)
        Sg, yg = g.rcs(l, 1e-3)
        low = np.tril(np.ones_like(So, dtype=bool))
        assert np.abs(Sg[low] - So[low]).max() <= 1e-10 * np.abs(So).max()
        assert np.abs(yg - yo).max() <= 1e-9 * np.abs(yo).max()


@pytest.mark.parametrize("points,opp", [(27, 4), (28, 4), (29, 6), (57, 24), (300, 24), (700, 4)])
@pytest.mark.parametrize("weighted", [False, True])
def test_reduced_camera_system(points, opp, weighted):
    rng = np.random.default_rng(points)
    prob = synth.tiny(seed=points, nx=6, ny=4, n_points=points, opp=opp, runs=[15, 9], spacing=0.5)
    if weighted:
        K = prob["obs_cam"].size
        a, c = rng.uniform(0.5, 2.0, K), rng.uniform(0.5, 2.0, K)
        prob["obs_winv"] = np.stack([a, 0.3 * np.sqrt(a * c), c], axis=1)
    prob, o, g = prepared(prob, 0)
    o.intersect()
    Xl, Wl = o.instance_state()
    o.set_instance_state(Xl + rng.normal(0, 0.02, Xl.shape), Wl)
    o.set_weights(np.where(rng.random(o.K) < 0.05, 1e-4, 1.0))
    sync_state(o, g)
    _check(o, g)


@pytest.mark.parametrize("points,track", [(40, 3.0), (60, 14.0)])
def test_reduced_camera_system_with_intrinsics(points, track):
    prob = synth.tiny_intrinsics(seed=points, n_cams=24, n_points=points, mean_track=track, n_sub=2)
    prob, o, g = prepared(prob, 0)
    o.intersect()
    _sync(o, g)
    _check(o, g)
