"""rpba_tune in the FP64 form times and chooses only what that form's kernels
read: not the CTA sizes of the linearisation and the intersection, which have
one launch shape each."""

import pytest

from paper_1910_08138_gb300 import rpba, synth

pytestmark = pytest.mark.gpu


def test_shapes_that_no_kernel_reads_are_not_timed():
    g = rpba.Rpba(synth.config(1), precision=0, solver=2, robust=1, robust_from_start=1)
    g.intersect()
    g.profile_enable(True)
    g.profile_select("k_exchange")  # counts launches, times none of these
    chosen = g.tune()
    prof, _ = g.profile_read()
    assert chosen["lin"] == 128 and chosen["isect"] == 128  # the defaults
    assert prof["k_linearize_f64"][0] == 1  # the assembly that the other timings need
    assert "k_isect_fused_d" not in prof
    assert prof["k_backsub_f64"][0] >= 15
    g.close()
