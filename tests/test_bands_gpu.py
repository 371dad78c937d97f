"""Multi-word gate on converged rollouts: pairs whose bounds leave a narrow band (rings of stripes,
every team width) or nothing at all, for patterns longer and shorter than their texts, in batches
small enough for a warp per pair and large enough for many pairs per warp."""
import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches, gate_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,K", [(3, 1024), (3, 1023), (3, 450), (260, 1022), (260, 190), (700, 70)])
@pytest.mark.parametrize("vocab", [20, 3000, 10 ** 9])
def test_converged_rollouts(G, K, vocab):
    rng = np.random.default_rng(7 * G + K)
    N, stride = 4, (K + 3) // 4 * 4
    base = rng.integers(0, vocab, size=(G, 1, stride)).astype(np.int32)
    seqs = np.broadcast_to(base, (G, N, stride)).copy()
    rate = rng.choice([0.0, 0.004, 0.03, 0.1, 0.3], size=(G, N, 1))
    edit = rng.random((G, N, stride)) < rate
    seqs[edit] = rng.integers(0, vocab, size=int(edit.sum()))
    for g in range(0, G, 3):                                 # an inserted run shifts the rest of one rollout
        at, by = int(rng.integers(1, K - 8)), int(rng.integers(1, 6))
        seqs[g, 0, at + by:] = seqs[g, 0, at:-by].copy()
    lens = np.where(rng.random((G, 1)) < 0.5, K, rng.integers(max(K - 40, 33), K + 1, size=(G, N))).astype(np.int32)
    lens[:: 7] = rng.integers(1, K + 1, size=lens[:: 7].shape)
    want = oracle.gate(seqs, lens, K, 0.12, threads=8)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.12), want, f"G={G} K={K} vocab={vocab}")
