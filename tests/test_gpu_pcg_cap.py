"""pcg_max_iter caps the CG steps that the refinement stages of the FP32 form's
PCG take when all sub-blocks go through them together, in every form of the
loop: a sub-block that converges early does not get steps that the slowest one
has used up. Blocks whose sub-blocks need very different numbers of steps.
"""

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba, synth
from test_gpu_pcg_solve_forms import _grid

pytestmark = pytest.mark.gpu


def _member(cams, seed):
    n = int(np.sqrt(cams))
    rng = np.random.Generator(np.random.PCG64(seed))
    return synth.grid_block(rng, n, cams // n, 4.0, 30.0, 25 * cams, 5, 0.5, 0.02, oblique_deg=30.0, nadir_every=5,
                            runs=[n * (cams // n)])


def _solve(prob, lm_step=False, **opts):
    g = rpba.Rpba(prob, precision=1, solver=1, robust=1, robust_from_start=1, max_inner=1, **opts)
    g.intersect()
    if lm_step:
        g.lm_step(1e-3)
    else:
        g.outer_iteration(robust=True)
    it, rr = g.solver_stats()
    out = it.copy(), g.solver_stages().copy(), rr.copy(), g.camera_rt()
    g.close()
    return out


# sub-blocks of 16 and 49 cameras: tiles in registers; 16 and 121: tiles read per step
@pytest.mark.parametrize("sizes", [(16, 49), (16, 121)])
def test_sub_blocks_stay_in_the_same_stage(sizes):
    prob = synth.merge_blocks([_member(c, 3 + k) for k, c in enumerate(sizes)])
    full = _solve(prob)
    assert np.all(full[1] >= 2) and np.all(full[2] <= 1e-8)
    mixed = 0
    for cap in range(1, int(full[0].max()) + 6):
        it, stages, rr, _ = _solve(prob, pcg_max_iter=cap)
        open_ = rr > 1e-8  # of a sub-block that has not converged
        assert np.all(stages[open_] == stages.max()), (cap, it, stages, rr)
        assert it.max() <= cap
        mixed += len(set(it)) > 1
    assert mixed  # some caps lay between the sub-blocks' counts


@pytest.mark.parametrize("sizes", [(16, 49), (16, 121)])
@pytest.mark.parametrize("lm_step", [False, True])
def test_one_kernel_stops_where_the_graph_nodes_stop(sizes, lm_step):
    """The same sub-blocks beside 160 of one camera (one CG step per stage), which
    a loop of graph nodes solves: the same steps and stages at every cap. LM steps
    outside a graph run that loop from the host, which counts up to a few idle
    steps towards the cap: there only caps that no stage reaches or all do."""
    members = [_member(c, 3 + k) for k, c in enumerate(sizes)]
    small, large = synth.merge_blocks(members), synth.merge_blocks(members + [_grid([1] * 160, 9)])
    n = sum(m["cam_pose"].shape[0] for m in members)
    slowest = int(_solve(small)[0].max())
    caps = {1, 2, 500} if lm_step else {1, 2, slowest // 3, slowest // 2, slowest - 3, slowest - 1, slowest,
                                        slowest + 1, 500}
    for cap in sorted(caps):
        a, b = _solve(small, lm_step, pcg_max_iter=cap), _solve(large, lm_step, pcg_max_iter=cap)
        np.testing.assert_array_equal(a[0], b[0][:len(sizes)], err_msg=str(cap))
        np.testing.assert_array_equal(a[1], b[1][:len(sizes)], err_msg=str(cap))
        np.testing.assert_allclose(a[3][:n], b[3][:n], rtol=0, atol=1e-9)
