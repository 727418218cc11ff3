"""A bounded wait of the direct solvers' kernels that runs out is an error of its
own (DEVICE_TIMEOUT), not a sub-block whose matrix is not positive definite: the
call ends, the state stays, and the context works on with a longer limit. The
limit of one look makes waits run out at once: an entry of the substitution
takes about a microsecond to arrive."""

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba, synth

pytestmark = pytest.mark.gpu

TIMEOUT, INVALID = 5, 1


# the substitution in FP64, in FP32, and behind the tensor-core factorisation
@pytest.mark.parametrize("opts", [dict(precision=0, solver=0), dict(precision=1, solver=2),
                                  dict(precision=1, solver=2, chol_tc=1)])
def test_a_wait_that_runs_out_is_reported(opts):
    prob = synth.tiny(seed=9, nx=99, ny=1, n_points=4000, opp=3, runs=[96, 3], spacing=2.0, oblique_deg=20,
                      nadir_every=2, extent=(-99.0, 99.0, -6.0, 6.0))
    g, h = rpba.Rpba(prob, **opts), rpba.Rpba(prob, **opts)
    for side in (g, h):
        side.intersect()
    before = g.camera_rt()
    g.set_wait_limit(0)
    for call in (g.bact, lambda: g.lm_step(1e-3), g.iterate):
        with pytest.raises(rpba.RpbaError) as e:
            call()
        assert e.value.status == TIMEOUT
        np.testing.assert_array_equal(g.camera_rt(), before)
    with pytest.raises(rpba.RpbaError) as e:
        g.set_wait_limit(-1)
    assert e.value.status == INVALID
    g.set_wait_limit(500_000_000)
    a, b = g.lm_step(1e-3), h.lm_step(1e-3)
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_allclose(a[3], b[3], rtol=0, atol=1e-6 * np.abs(b[3]).max())
    g.bact()
    for side in (g, h):
        side.close()
