"""Batches whose pairs are run from both ends: edges of the blocks a lane holds (16 and 32 lanes of 32 rows, one
past them), texts of one to five columns, chains of occurrences, group sizes around a cluster's, and the sizes at
which a group's CTAs stop naming its symbols themselves."""
import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches, gate_gpu


def _batch(rng, G, N, K, vocab):
    stride = (K + 3) // 4 * 4
    lens = np.minimum(K, rng.choice([1, 2, 3, 4, 5, 31, 32, 33, K // 2, K - 3, K - 2, K - 1, K], size=(G, N))).astype(np.int32)
    lens[:, 0] = K
    seqs = np.zeros((G, N, stride), dtype=np.int32)
    for g in range(G):
        base = rng.integers(0, vocab, size=stride)
        for i in range(N):
            row = np.where(rng.random(stride) < (0.2 if g % 2 else 0.9), rng.integers(0, vocab, size=stride), base)
            seqs[g, i, :lens[g, i]] = row[:lens[g, i]]
    return seqs, lens


@pytest.mark.gpu
@pytest.mark.parametrize("G,N,K,vocab", [
    (3, 8, 33, 4), (3, 8, 64, 30), (2, 8, 65, 30), (9, 8, 288, 90), (9, 8, 512, 170), (3, 8, 513, 30), (4, 4, 1021, 400),
    (4, 3, 1024, 340), (5, 2, 1024, 1 << 30), (3, 9, 100, 30), (2, 17, 250, 80), (1, 32, 500, 200), (40, 8, 48, 10),
])
def test_gate_from_both_ends(G, N, K, vocab):
    rng = np.random.default_rng(G * K + N)
    seqs, lens = _batch(rng, G, N, K, vocab)
    for norm, thr in ((0, 0.5), (1, 0.5 * K)):
        want = oracle.gate(seqs, lens, K, thr, norm, threads=8)
        assert_gate_matches(gate_gpu(seqs, lens, K, thr, norm), want, f"G={G} N={N} K={K} norm={norm}")


@pytest.mark.gpu
@pytest.mark.parametrize("N,K", [(8, 48), (8, 600), (12, 48)])
def test_negative_lengths_are_reported(N, K):
    rng = np.random.default_rng(K)
    seqs, lens = _batch(rng, 4, N, K, 50)
    lens[2, 1] = -5
    status = []
    got = gate_gpu(seqs, lens, K, 0.5, 0, status=status)
    assert status == [1]
    assert_gate_matches(got, oracle.gate(seqs, np.maximum(lens, 0), K, 0.5, 0, threads=8), f"N={N} K={K}")


@pytest.mark.gpu
@pytest.mark.parametrize("G,N,K,vocab", [(2, 17, 254, 80), (1, 18, 254, 80), (2, 20, 513, 150), (1, 32, 1024, 340), (4, 32, 300, 100), (5, 32, 300, 100), (3, 18, 253, 80)])
def test_more_texts_than_warps(G, N, K, vocab):
    """Patterns with up to sixteen texts: a warp for each while every CTA has an SM, eight warps in turns beyond that."""
    rng = np.random.default_rng(G * K + N)
    seqs, lens = _batch(rng, G, N, K, vocab)
    want = oracle.gate(seqs, lens, K, 0.5, 0, threads=8)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.5, 0), want, f"G={G} N={N} K={K}")
