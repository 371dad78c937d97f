"""Groups of eight on either side of the sizes between which a CTA's pair states come by asynchronous copies: drawn groups,
the first and the last of them equal to the oracle on the prefixes so far."""
import numpy as np
import pytest

import oracle
from helpers import IncrementalGate, assert_gate_matches


@pytest.mark.gpu
@pytest.mark.parametrize("G", [16785, 16786, 46428, 46429])
def test_groups_of_eight(G):
    N, steps = 8, 6
    rng = np.random.default_rng(G)
    actions = rng.integers(0, rng.choice([3, 40], size=(G, 1)), size=(steps, G, N))
    actions = np.where(rng.random((steps, G, N)) < 0.1, -2 ** 31, actions).astype(np.int32)
    check = np.unique(np.concatenate([rng.integers(0, G, 200), [0, G - 2, G - 1]]))
    gate = IncrementalGate(G, N, steps)
    seqs, lens = np.zeros((len(check), N, 32), dtype=np.int32), np.zeros((len(check), N), dtype=np.int32)
    for t in range(steps):
        got = gate.step(actions[t], 0.4)
        g, i = np.nonzero(actions[t][check] != -2 ** 31)
        seqs[g, i, lens[g, i]] = actions[t][check][g, i]
        lens[g, i] += 1
        assert_gate_matches(tuple(x[check] for x in got), oracle.gate(seqs, lens, 32, 0.4, threads=8), f"G={G} step {t + 1}")
