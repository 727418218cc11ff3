"""The FP32 form's CG loop on the device in its three forms: one kernel with
the tiles in registers (sub-blocks of up to 64 tiles), one kernel with 32 warps
per CTA (larger ones), and conditional graph nodes (many sub-blocks). Each
against the host-driven loop of the single kernels, which does the same
arithmetic in the same order: the same CG steps and refinement stages of every
sub-block, and the same state up to the order of the Schur kernel's FP64
atomics (the tolerance of test_gpu_pcg_device_loop.py). Sub-blocks of uneven
size, one of a single camera; without and with per-camera intrinsics.
"""

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba, synth

pytestmark = pytest.mark.gpu


def _grid(runs, seed):
    n = sum(runs)
    nx = int(np.ceil(np.sqrt(n)))
    rng = np.random.Generator(np.random.PCG64(seed))
    return synth.grid_block(rng, nx, int(np.ceil(n / nx)), 4.0, 30.0, 25 * n, 5, 0.5, 0.02, oblique_deg=30.0,
                            nadir_every=5, n_cams=n, runs=runs)


BLOCKS = {
    "registers": lambda: _grid([1, 5, 6, 27, 53], 1),
    "wide": lambda: _grid([120, 54, 1], 2),
    "nodes": lambda: _grid([3] * 150 + [1, 2, 4, 8], 3),
    "registers_k1": lambda: synth.tiny_intrinsics(seed=1, n_cams=60, n_points=1500, n_sub=2),
    "wide_k1": lambda: synth.tiny_intrinsics(seed=2, n_cams=140, n_points=3000, n_sub=2),
}


def _run(prob, host_loop):
    g = rpba.Rpba(prob, precision=1, solver=1, robust=1, robust_from_start=1, max_inner=1)
    g.intersect()
    if host_loop:  # a loop kernel that is timed runs on its own, from the host
        g.profile_enable(True)
        g.profile_select("k_pcg_symv32")
    out = []
    for _ in range(2):
        g.outer_iteration(robust=True)
        it, rr = g.solver_stats()
        out.append((it.copy(), g.solver_stages().copy(), g.camera_rt(), rr.copy()))
    g.close()
    return out


@pytest.mark.parametrize("name", list(BLOCKS))
def test_device_loop_forms_equal_the_host_loop(name):
    prob = BLOCKS[name]()
    for d, h in zip(_run(prob, False), _run(prob, True)):
        np.testing.assert_array_equal(d[0], h[0])
        np.testing.assert_array_equal(d[1], h[1])
        assert np.all(d[1] >= 1)
        np.testing.assert_allclose(d[2], h[2], rtol=0, atol=1e-9)
        np.testing.assert_allclose(d[3], h[3], rtol=1e-3, atol=1e-12)
