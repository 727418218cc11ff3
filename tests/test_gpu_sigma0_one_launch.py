"""rpba_sigma0_noalloc at the edges of its CTAs, in calls of changing size.

The sums are of K non-negative terms added in a tree: relative error below
1e-13. A residual is the difference of image coordinates near 1000 pixels, so it
carries an absolute error near 1e-12; for a sum of a single residual as small as
1e-3 pixels that is 2e-9 of its square. Bound: 1e-8 for the squares, the counts
exactly.
"""

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(1, 1), (256, 256), (255, 257), (257, 1)], [(70_001, 9_000), (1, 1), (512, 513)],
                                   [(300_000, 70_000), (300_000, 70_000)]])
@pytest.mark.parametrize("options", [False, True])
def test_sums_match_numpy(sizes, options):
    import torch
    rng = np.random.default_rng(5)
    M = 7
    R, _ = np.linalg.qr(np.eye(3) + 0.05 * rng.normal(size=(M, 3, 3)))
    R = R * np.sign(np.einsum("mii->mi", R))[:, None, :]
    t = np.stack([rng.normal(0, 2, M), rng.normal(0, 2, M), rng.uniform(25, 35, M)], axis=1)
    intr = np.tile([1000.0, 1000.0, 750.0], (M, 1))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    for K, N in sizes:
        X = rng.normal(0, 3, (N, 3))
        cam, pt = rng.integers(0, M, K).astype(np.int32), rng.integers(0, N, K).astype(np.int32)
        xc = np.einsum("kab,kb->ka", R[cam], X[pt]) + t[cam]
        r = rng.normal(0, 0.5, (K, 2))
        xy = 1000.0 * xc[:, :2] / xc[:, 2:] + intr[cam, 1:] - r
        active, w, W = np.ones(N, np.uint8), np.ones(K), np.tile([1.0, 0.0, 1.0], (K, 1))
        if options:
            active = (rng.random(N) < 0.9).astype(np.uint8)
            w = np.where(rng.random(K) < 0.1, 1e-4, 1.0)
            W = np.stack([rng.uniform(0.5, 2, K), rng.uniform(-0.2, 0.2, K), rng.uniform(0.5, 2, K)], axis=1)
        on = active[pt] == 1
        q = w * (W[:, 0] * r[:, 0] ** 2 + 2 * W[:, 1] * r[:, 0] * r[:, 1] + W[:, 2] * r[:, 1] ** 2)
        one = on & (w == 1.0)
        want = [q[on].sum(), on.sum(), (r[one] ** 2).sum(), one.sum(), active.sum()]
        a = [dev(v) for v in (R, t, intr, X)]
        opt = [dev(v) for v in (active, W, w)] if options else [None] * 3
        o = [dev(v) for v in (cam, pt, xy)]
        ptr = lambda v: None if v is None else v.data_ptr()
        s0, rms, sums = rpba.rpba_sigma0_noalloc(M, N, K, *map(ptr, a), ptr(opt[0]), *map(ptr, o), ptr(opt[1]),
                                                 ptr(opt[2]), stream=torch.cuda.current_stream())
        np.testing.assert_allclose(sums[[0, 2]], np.array(want)[[0, 2]], rtol=1e-8, atol=0)
        assert list(sums[[1, 3, 4]]) == [want[1], want[3], want[4]]
