"""Large batches of short prefixes in groups of four and five, whose patterns have two warps each, on either side of the length from
which less frequent symbols get the mask rows that others leave; vocabularies that exceed the rows by a few and by many symbols."""
import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches, gate_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,G", [(4, 33, 2000), (5, 64, 1300), (4, 96, 1800), (4, 97, 1800), (5, 128, 1100), (5, 129, 1100), (4, 256, 1300)])
def test_patterns_of_two_warps(N, K, G):
    import torch
    import paper_2605_05802_b200 as sr
    rng = np.random.default_rng(K + G)
    unique, stride = 80, (K + 3) // 4 * 4
    vocab = np.array([3, K // 8, K // 3, K, 3 * K])[np.arange(unique) % 5].reshape(-1, 1, 1)
    base, own = (rng.integers(0, vocab, size=(unique, n, stride)) for n in (1, N))
    rate = np.array([0.01, 0.05, 0.3])[np.arange(unique) % 3].reshape(-1, 1, 1)
    some = np.where(rng.random(own.shape) < rate, own, base).astype(np.int32)
    some_lens = np.full((unique, N), K, dtype=np.int32)
    some_lens[::4] = rng.integers(0, K + 1, size=some_lens[::4].shape)
    which = rng.integers(0, unique, size=G)
    want = tuple(x[which] for x in oracle.gate(some, some_lens, K, 0.12, threads=8))
    seqs, lens = some[which], some_lens[which]
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.12), want, f"G={G} N={N} K={K}")
    stop = torch.empty(G, dtype=torch.uint8, device="cuda")
    ws = torch.empty(sr.sr_gate_workspace_bytes(G, N, stride, K), dtype=torch.uint8, device="cuda")
    sr.sr_gate_decide(torch.from_numpy(seqs).cuda(), torch.from_numpy(lens).cuda(), K, 0.12, stop=stop, workspace=ws)
    assert np.array_equal(stop.cpu().numpy(), want[3])
