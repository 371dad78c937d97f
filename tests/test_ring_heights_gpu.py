"""Rings of every height: bands at the widths at which a ring of so many lanes and blocks just holds them, or just does not, in
batches large enough that few lanes with high stripes are cheapest, and whose tasks outnumber the warps of the recurrence."""
import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches, gate_gpu

pytestmark = pytest.mark.gpu


def limits(T):
    """First widths that rings of T lanes of one to four blocks do not hold: w + 32 R + 3 + 8 a < T (32 R + 4)."""
    return [T * (32 * R + 4) - 32 * R - 3 - 8 * (2 if R <= 2 else 1) for R in (1, 2, 3, 4)]


# Substitutions by symbols that both prefixes hold leave a band of as many diagonals.  2, 4 and 8 lanes a pair: 16, 8 and 4 pairs to a task.
@pytest.mark.parametrize("T,N,K,G", [(2, 2, 600, 45000), (2, 2, 333, 90000), (4, 2, 1024, 24000), (4, 2, 900, 44000), (8, 2, 1021, 11000), (8, 3, 1024, 8000)])
def test_bands_at_the_limits_of_rings_of_every_height(T, N, K, G):
    rng = np.random.default_rng(K + G)
    widths = [w + d for w in limits(T) for d in (-2, -1, 0, 1) if 2 <= w + d < K * 2 // 3]
    unique, stride = 16 * len(widths), (K + 3) // 4 * 4
    some = np.zeros((unique, N, stride), dtype=np.int32)
    some[:] = rng.integers(0, K // 8, size=(unique, 1, stride))
    for u in range(unique):
        for i in range(1, N):
            at = rng.choice(K - 1, size=widths[u % len(widths)], replace=False)
            some[u, i, at] = (some[u, i, at] + rng.integers(1, K // 8, size=at.size)) % (K // 8)
    lens = np.full((unique, N), K, dtype=np.int32)
    lens[unique * 3 // 4:] = rng.integers(K - 30, K + 1, size=lens[unique * 3 // 4:].shape)
    which = rng.integers(0, unique, size=G)
    want = oracle.gate(some, lens, K, 0.12, threads=8)
    assert_gate_matches(gate_gpu(some[which], lens[which], K, 0.12), tuple(x[which] for x in want), f"G={G} N={N} K={K}")
