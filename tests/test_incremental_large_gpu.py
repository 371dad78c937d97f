"""Incremental gate on batches large enough for the thread-per-rollout kernel: every width of its mask
loop, more and fewer pairs than threads in a CTA, pauses, early ends and full rollouts."""
import numpy as np
import pytest

import oracle
from helpers import IncrementalGate, assert_gate_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,max_steps", [(4, 9), (5, 6), (8, 32), (9, 5), (17, 5), (32, 4)])
def test_large_batches(N, max_steps):
    P = N * (N - 1) // 2
    G = 550000 // P + 5
    rng = np.random.default_rng(N)
    steps = max_steps + 1                                    # the last action finds full rollouts
    vocab = rng.choice([3, 40, 4096], size=(G, 1))
    actions = rng.integers(0, 1 << 30, size=(steps, G, N)) % vocab
    actions = np.where(rng.random((steps, G, N)) < 0.1, -2 ** 31, actions).astype(np.int32)
    check = np.unique(np.concatenate([rng.integers(0, G, 300), [0, 1, G - 2, G - 1]]))
    gate = IncrementalGate(G, N, max_steps)
    seqs = np.zeros((len(check), N, 32), dtype=np.int32)
    lens = np.zeros((len(check), N), dtype=np.int32)
    for t in range(steps):
        got = gate.step(actions[t], 0.4)
        a = actions[t][check]
        g, i = np.nonzero((a != -2 ** 31) & (lens < max_steps))
        seqs[g, i, lens[g, i]] = a[g, i]
        lens[g, i] += 1
        if t % 4 == 0 or t >= steps - 2:
            want = oracle.gate(seqs, lens, max_steps, 0.4, threads=8)
            assert_gate_matches(tuple(x[check] for x in got), want, f"N={N} step {t + 1}")
