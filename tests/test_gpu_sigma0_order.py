"""rpba_sigma0_noalloc from two host threads: calls whose work does not overlap
on the GPU give their own sums, whichever of them was entered first."""

import threading
import time

import numpy as np
import pytest

from paper_1910_08138_gb300 import rpba

pytestmark = pytest.mark.gpu


def _block(n_points, seed):
    import torch
    rng = np.random.default_rng(seed)
    K = 4 * n_points
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    arrays = [dev(np.eye(3).reshape(1, 9)), dev(np.array([[0.0, 0.0, 30.0]])), dev(np.array([[1000.0, 500.0, 500.0]])),
              dev(rng.normal(size=(n_points, 3))), None, dev(np.zeros(K, np.int32)),
              dev(rng.integers(0, n_points, K).astype(np.int32)), dev(rng.normal(500, 30, (K, 2)))]
    return (1, n_points, K, *[None if a is None else a.data_ptr() for a in arrays]), arrays


@pytest.mark.parametrize("sizes", [(3000, 3000), (3000, 500), (10, 40_000)])
def test_a_call_that_waits_on_its_stream_gets_its_own_sums(sizes):
    import torch
    (early, _a), (late, _b) = _block(sizes[0], 1), _block(sizes[1], 2)
    want = [rpba.rpba_sigma0_noalloc(*c)[2] for c in (early, late)]
    assert want[0][0] != want[1][0]
    waiting, other = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(2):  # a count left over would show in the next round
        got = [None, None]
        torch.cuda.synchronize()
        with torch.cuda.stream(waiting):
            torch.cuda._sleep(1_000_000_000)  # about 0.5 s: the call below is entered, its work waits

        def call():
            got[0] = rpba.rpba_sigma0_noalloc(*early, stream=waiting)[2]

        t = threading.Thread(target=call)
        t.start()
        time.sleep(0.05)
        got[1] = rpba.rpba_sigma0_noalloc(*late, stream=other)[2]
        assert got[0] is None  # the first call is still waiting
        t.join()
        for g, w in zip(got, want):
            np.testing.assert_array_equal(g, w)
