"""The direct solves of the reduced camera system at the edges of their 32-row
tiles: sub-blocks of 1 to 43 cameras (6 to 258 unknowns, 1 to 9 tiles, with
and without padding), two sub-blocks of different size per block. The solution
of one LM step against the RCS of the same state (rpba_rcs): backward error
||S dC - y|| / (||S|| ||dC|| + ||y||). A Cholesky solve in FP64 is backward
stable, n eps times a small constant: 300 x 1.1e-16 x 10 < 1e-12 (solver 0).
Solver 2 refines its FP32 solve twice with an FP64 residual: below its FP32
error, 300 x 6e-8 x 10 = 2e-4, squared at least once, 1e-7.
"""

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver,tol", [(0, 1e-12), (2, 1e-7)])
@pytest.mark.parametrize("cams", [1, 5, 6, 11, 16, 43])
def test_direct_solve_of_tile_edges(cams, solver, tol):
    other = 3
    prob = synth.tiny(seed=cams, nx=cams + other, ny=1, n_points=60 * (cams + other), opp=3, runs=[cams, other],
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
