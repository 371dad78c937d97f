"""Pairs whose band just fits a ring of stripes, or just does not: K substitutions by symbols that both prefixes hold leave a
band of K + 1 diagonals.  Batches with fewer tasks than warps, whose tasks are dealt out, and with more."""
import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches, gate_gpu

pytestmark = pytest.mark.gpu

# T lanes of R blocks follow a band of w + 1 diagonals where w + 32 R + 3 + 8 a < T (32 R + 4), a = 2 for R <= 2 and 1 above
LIMITS = sorted({T * (32 * R + 4) - 32 * R - 3 - 8 * (2 if R <= 2 else 1) for T in (2, 4, 8) for R in (1, 2, 3, 4)})


@pytest.mark.parametrize("G,N,K", [(720, 2, 1024), (2600, 2, 700), (730, 2, 1021)])
def test_bands_at_the_limits_of_rings(G, N, K):
    rng = np.random.default_rng(K + G)
    widths = np.array([w + d for w in LIMITS for d in (-2, -1, 0, 1) if 2 <= w + d < K // 2])
    stride = (K + 3) // 4 * 4
    seqs = np.zeros((G, N, stride), dtype=np.int32)
    for g in range(G):
        base = rng.integers(0, 2 ** 31 - 1, size=stride, dtype=np.int32)
        repeats = rng.integers(0, stride, size=stride // 8)              # symbols with mask rows
        base[repeats] = base[rng.integers(0, stride, size=repeats.size)]
        seqs[g] = base
        for i in range(1, N):                                           # substitutions against rollout 0
            at = rng.choice(K - 1, size=int(rng.choice(widths)), replace=False)
            seqs[g, i, at] = seqs[g, 0, (at + 1 + rng.integers(0, K - 1, size=at.size)) % K]
    lens = np.full((G, N), K, dtype=np.int32)
    lens[::3] = rng.integers(K - 30, K + 1, size=lens[::3].shape)
    want = oracle.gate(seqs, lens, K, 0.12, threads=8)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.12), want, f"G={G} N={N} K={K}")
