"""Pairs settled from their few matches: vocabularies from which two prefixes have about as many symbols in
common as a warp has lanes, with and without repeated symbols, on batches that are large enough to be sorted
into warp tasks and on small ones."""
import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches, gate_gpu


def _batch(rng, G, N, K, vocab):
    """A third of the groups converged, a third with a shared head, a third shifted against each other."""
    stride = (K + 3) // 4 * 4
    lens = rng.integers(1, K + 1, size=(G, N)).astype(np.int32)
    lens[:, 0] = K
    seqs = np.zeros((G, N, stride), dtype=np.int32)
    for g in range(G):
        base = rng.integers(0, vocab, size=2 * stride)
        head = int(rng.integers(0, K + 1))
        for i in range(N):
            own = rng.integers(0, vocab, size=stride)
            if g % 3 == 0:
                row = np.where(rng.random(stride) < 0.1, own, base[:stride])
            elif g % 3 == 1:
                row = np.where(np.arange(stride) < head, base[:stride], own)
            else:
                at = int(rng.integers(0, 3))
                row = np.where(rng.random(stride) < 0.3, own, base[at:at + stride])
            seqs[g, i, :lens[g, i]] = row[:lens[g, i]]
    return seqs, lens


@pytest.mark.gpu
@pytest.mark.parametrize("G,N,K,vocab", [
    (38, 16, 1024, 150000),     # sorted batches: 7 matches a pair of unrelated rollouts
    (38, 16, 1021, 33000),      # 31 of them: about as many as there are lanes; repeated symbols everywhere
    (84, 16, 257, 3000),        # 22, and a text's last quad of one column
    (6, 8, 1024, 33000),        # a warp for every pair
    (5, 5, 640, 20000),
])
def test_gate_with_few_matches(G, N, K, vocab):
    rng = np.random.default_rng(vocab + K)
    seqs, lens = _batch(rng, G, N, K, vocab)
    want = oracle.gate(seqs, lens, K, 0.4, 0, threads=8)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.4, 0), want, f"G={G} N={N} K={K} vocab={vocab}")


def _recurring_heads(rng, G, N, K):
    """Groups that share a head of 200 symbols and more; the tails of every other rollout take up to thirty symbols of the
    head again, which so occur once in the patterns of the others, before the place where the pair begins to differ."""
    stride = (K + 3) // 4 * 4
    lens = rng.integers(K // 2, K + 1, size=(G, N)).astype(np.int32)
    lens[:, 0] = K
    seqs = np.zeros((G, N, stride), dtype=np.int32)
    for g in range(G):
        head = min(int(rng.integers(200, 901)), K - 40)
        symbols = rng.choice(1 << 20, size=stride * (N + 1), replace=False)
        for i in range(N):
            row = np.concatenate([symbols[:head], symbols[stride * (i + 1):stride * (i + 2) - head]])
            if i % 2:
                again = min(int(rng.integers(1, 31)), stride - head)
                row[head + rng.choice(stride - head, size=again, replace=False)] = symbols[rng.choice(head, size=again, replace=False)]
            seqs[g, i, :lens[g, i]] = row[:lens[g, i]]
    return seqs, lens


@pytest.mark.gpu
@pytest.mark.parametrize("G,N,K", [(41, 16, 1024), (41, 16, 1001), (6, 8, 1024), (5, 5, 997), (12, 8, 400)])
def test_symbols_of_the_common_prefix_that_come_again(G, N, K):
    rng = np.random.default_rng(G * K)
    seqs, lens = _recurring_heads(rng, G, N, K)
    want = oracle.gate(seqs, lens, K, 0.4, 0, threads=8)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.4, 0), want, f"G={G} N={N} K={K}")


@pytest.mark.gpu
@pytest.mark.parametrize("G,N,K,vocab", [(2200, 8, 48, 3000), (1500, 8, 100, 400), (1500, 8, 100, 100000), (5000, 2, 256, 3000), (60, 16, 256, 3000)])
def test_short_prefixes_with_few_matches(G, N, K, vocab):
    """Some of a batch's pairs listed and some left to the recurrence: about where one costs as much as the other."""
    rng = np.random.default_rng(vocab + K)
    seqs, lens = _batch(rng, G, N, K, vocab)
    want = oracle.gate(seqs, lens, K, 0.4, 0, threads=8)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.4, 0), want, f"G={G} N={N} K={K} vocab={vocab}")
