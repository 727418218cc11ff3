"""Loss and gradient of the preconditioner's network at the edges of its kernels:
probe counts around the groups of 4, systems around the 5-node tiles, node counts
around the 8- and 16-node CTAs, and a set large enough for a CTA to take several
chunks. Bounds as in test_gnn_gpu.py (FP32 activations: 1e-5 for the loss, 1e-3 for
gradients). Copies of one system have that system's loss and gradient; both sides
are FP32 sums of the same terms: 1e-4."""

import numpy as np
import pytest

from oracle import gnn
from paper_1910_08138_gb300 import rpba, synth
from test_gnn_gpu import _as_applied, _trainer

pytestmark = pytest.mark.gpu


def _weights(n):
    return (np.random.default_rng(8).normal(size=n) * 0.1).astype(np.float32)


@pytest.mark.parametrize("sizes,probes", [((4,), 1), ((5, 6), 2), ((8,), 3), ((16, 11), 4), ((17, 4), 5), ((10, 15), 9)])
def test_matches_oracle(sizes, probes):
    sy = synth.rcs_like_systems(3, sizes=sizes, n_probes=probes)
    gs = [(gnn.graph(S, S.shape[0] // 6), z) for S, z in sy]
    G = _trainer(sy)
    w = _weights(G.n_params)
    G.set_weights(w)
    loss, grad = G.loss_grad()
    lo, go = gnn.loss_and_grad(_as_applied(w), gs)
    assert loss == pytest.approx(lo, rel=1e-5, abs=1e-5)
    assert np.linalg.norm(grad - go) <= 1e-3 * np.linalg.norm(go)


def test_chunks_of_one_cta():
    sy = synth.rcs_like_systems(4, sizes=(23,), n_probes=2)
    one, many = _trainer(sy), _trainer(sy * 230)  # 5290 nodes: two per-CTA chunks for some
    w = _weights(one.n_params)
    one.set_weights(w)
    many.set_weights(w)
    (l1, g1), (lm, gm) = one.loss_grad(), many.loss_grad()
    assert lm == pytest.approx(l1, rel=1e-10)
    assert np.linalg.norm(gm - g1) <= 1e-4 * np.linalg.norm(g1)
