"""Multi-word gate on prefixes whose symbols occur several times: mask rows, the occurrence
count from which a symbol gets one, the chains of the others, and common prefixes of such pairs."""
import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches, gate_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [33, 64, 500, 1024])
@pytest.mark.parametrize("times", [2, 3, 4, 7, 8, 60])
def test_symbols_with_a_given_number_of_occurrences(K, times):
    rng = np.random.default_rng(1000 * K + times)
    G, N, stride = 6, 5, (K + 3) // 4 * 4
    pool = np.arange(stride) // times                       # every symbol `times` times ...
    seqs = np.stack([[rng.permutation(pool) for _ in range(N)] for _ in range(G)]).astype(np.int32)
    seqs[1] += rng.integers(0, 40000, size=(N, stride)) * (rng.random((N, stride)) < 0.5)   # ... or some of them once
    seqs[2:5, :, : K // 2] = seqs[2:5, :1, : K // 2]        # common prefixes
    seqs[4, :, 31] += np.arange(N)                          # ... that end around a word boundary
    seqs[5] = seqs[5, :1]
    lens = rng.integers(K // 3, K + 1, size=(G, N)).astype(np.int32)
    lens[0] = K
    want = oracle.gate(seqs, lens, K, 0.4, threads=8)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.4), want, f"K={K}, {times} occurrences")


@pytest.mark.parametrize("K", [64, 300, 1024])
def test_symbols_that_crowd_one_slot_of_the_table(K):
    """IDs chosen so that dozens of them hash to one slot under the first hash: many rounds until all have names."""
    rng = np.random.default_rng(K)
    inverse = pow(0x9E3779B1, -1, 1 << 32)
    crowd = (np.array([5 << 25], dtype=np.uint64) + np.arange(40, dtype=np.uint64)) * np.uint64(inverse) % np.uint64(1 << 32)
    crowd = crowd.astype(np.uint32).view(np.int32)
    G, N, stride = 5, 6, (K + 3) // 4 * 4
    seqs = rng.integers(-2 ** 31, 2 ** 31, size=(G, N, stride)).astype(np.int32)
    pick = rng.random((G, N, stride)) < np.array([0.05, 0.3, 0.9, 0.9, 0.5]).reshape(G, 1, 1)
    seqs[pick] = rng.choice(crowd, size=int(pick.sum()))
    seqs[3, 1:] = np.where(rng.random((N - 1, stride)) < 0.1, seqs[3, 1:], seqs[3, :1])
    lens = rng.integers(K // 2 + 1, K + 1, size=(G, N)).astype(np.int32)
    want = oracle.gate(seqs, lens, K, 0.4, threads=8)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.4), want, f"K={K}")


@pytest.mark.parametrize("N,K", [(2, 33), (3, 128), (2, 129), (5, 256), (4, 257), (6, 384), (2, 385), (9, 40), (10, 513), (3, 641),
                                 (13, 60), (15, 70), (16, 769), (2, 897), (17, 130)])
def test_every_number_of_warps_per_pattern(N, K):
    """The per-pattern pass has a warp for every 128 positions and for every text: one to eight."""
    rng = np.random.default_rng(100 * N + K)
    G, stride = 7, (K + 3) // 4 * 4
    seqs = np.where(rng.random((G, N, stride)) < 0.2, rng.integers(0, 60, size=(G, N, stride)), rng.integers(0, 10 ** 6, size=(G, N, stride)))
    seqs[1::2] = np.where(rng.random((3, N, stride)) < 0.8, seqs[1::2, :1], seqs[1::2])
    lens = rng.integers(0, K + 1, size=(G, N)).astype(np.int32)
    lens[::2] = K
    seqs = seqs.astype(np.int32)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.4), oracle.gate(seqs, lens, K, 0.4, threads=8), f"N={N} K={K}")


@pytest.mark.parametrize("N,G", [(4, 6), (2, 2600)])        # computed in the CTAs of the patterns; sorted into warp tasks
@pytest.mark.parametrize("K", [40, 200, 1024])
def test_rows_left_by_frequent_symbols_go_to_others(N, G, K):
    """Patterns whose repeated symbols just fit the pool of mask rows or exceed it by a few or many, with occurrences of two to
    five mixed: frequent ones have rows, others take what is left, the last ones are chains."""
    rng = np.random.default_rng(K + G)
    cap, stride = (K + 7) // 8, (K + 3) // 4 * 4
    seqs = np.empty((G, N, stride), dtype=np.int32)
    for g in range(G if G < 100 else 40):
        often = [0, 1, cap - 1, cap, cap + 1][g % 5]          # symbols of three to five occurrences, and of two
        times = np.concatenate([rng.integers(3, 6, size=often), np.full(max(cap + [-1, 0, 1, 3, cap][g % 7 % 5] - often, 0), 2)])
        times = times[np.cumsum(times) <= K]
        pool = np.concatenate([np.repeat(np.arange(times.size), times), 10 ** 6 + np.arange(stride)])[:stride]
        for i in range(N):
            seqs[g, i] = rng.permutation(pool[:stride])
        seqs[g, 1:, : K // 3] = np.where(rng.random((N - 1, K // 3)) < 0.9, seqs[g, :1, : K // 3], seqs[g, 1:, : K // 3])
    for g in range(40, G):
        seqs[g] = seqs[g % 40]
    lens = np.full((G, N), K, dtype=np.int32)
    lens[::3] = rng.integers(K - 7, K + 1, size=lens[::3].shape)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.4), oracle.gate(seqs, lens, K, 0.4, threads=8), f"G={G} N={N} K={K}")
