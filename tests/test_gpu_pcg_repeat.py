"""The FP32 form's block-Jacobi PCG gives the same bits in every call from the
same state, and in every form of its loop (one kernel with the tiles in
registers or read per step, conditional graph nodes, host-driven): no sum that
decides a rounding depends on the order in which CTAs arrive."""

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba
from test_gpu_pcg_solve_forms import BLOCKS, _grid, _run

pytestmark = pytest.mark.gpu


def _passes(prob, n):
    g = rpba.Rpba(prob, precision=1, solver=1, robust=1, robust_from_start=1, max_inner=1)
    out = []
    for _ in range(n):
        g.set_cameras(prob["cam_pose"])
        g.set_points(prob["points"], np.ones(g.N, np.uint8))
        g.intersect()
        g.iterate(1)
        out.append(np.concatenate([g.cameras().ravel(), g.points()[0].ravel()]))
    g.close()
    return np.array(out)


@pytest.mark.parametrize("name", ["wide", "nodes"])
def test_repeated_calls_have_the_same_bits(name):
    prob = _grid([125] * 8, 5) if name == "wide" else BLOCKS[name]()
    a, b = _passes(prob, 40), _passes(prob, 40)
    np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("name", list(BLOCKS))
def test_forms_of_the_loop_have_the_same_bits(name):
    prob = BLOCKS[name]()
    for d, h in zip(_run(prob, False), _run(prob, True)):
        for x, y in zip(d, h):
            np.testing.assert_array_equal(x, y)
