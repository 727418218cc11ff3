"""The substitution of the direct solves where its ring of 16 steps wraps and
where a CTA owns more tiles than it holds in registers: sub-blocks of 15 to 36
tiles (80 to 190 cameras) beside a small one. Backward error of the step's
solution against the RCS of the same state, as in test_gpu_rcs_solve.py: n eps
times a small constant, 1140 x 1.1e-16 x 10 = 1.3e-12 (solver 0: 2e-12); FP32 with
two refinements, (1140 x 6e-8 x 10)^2 = 4.7e-7 (solver 2: 1e-6).
"""

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver,tol", [(0, 2e-12), (2, 1e-6)])
@pytest.mark.parametrize("cams", [80, 86, 96, 171, 190])
def test_substitution_of_many_tiles(cams, solver, tol):
    other = 3
    prob = synth.tiny(seed=cams, nx=cams + other, ny=1, n_points=40 * (cams + other), opp=3, runs=[cams, other],
                      spacing=2.0, oblique_deg=20, nadir_every=2, extent=(-cams - 3.0, cams + 3.0, -6.0, 6.0))
    g = rpba.Rpba(prob, precision=1 if solver == 2 else 0, solver=solver)
    g.intersect()
    lam = 1e-3
    systems = [g.rcs(l, lam) for l in range(g.L)]
    acc, _, _, dc, _ = g.lm_step(lam)
    off = 0
    for l, (S, y) in enumerate(systems):
        x = dc[off:off + y.size]
        off += y.size
        assert acc[l] >= 0
        err = np.linalg.norm(S @ x - y) / (np.linalg.norm(S, 2) * np.linalg.norm(x) + np.linalg.norm(y))
        assert err <= tol, (l, err)
    g.close()
