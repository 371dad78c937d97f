"""The mask alone for batches of more than 1024 pairs over the line for pairs from both ends, whose mask rows are made after the bounds
for the groups that these leave open: one pattern a group, odd and even groups, next to prefixes that are too short for it."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,N,K,vocab", [(1100, 2, 600, 300), (5000, 2, 257, 60), (500, 3, 400, 100), (700, 4, 300, 30), (200, 5, 520, 2000),
                                         (230, 7, 700, 90), (1100, 2, 1024, 500), (120, 11, 260, 70), (60, 16, 1000, 3000), (900, 5, 256, 40)])
def test_mask_alone_of_large_batches(G, N, K, vocab):
    import torch
    import paper_2605_05802_b200 as sr
    rng = np.random.default_rng(G + K)
    stride = (K + 3) // 4 * 4
    base = rng.integers(0, vocab, size=(G, 1, stride))
    rate = rng.random((G, 1, 1)) * 0.4
    seqs = np.where(rng.random((G, N, stride)) < rate, rng.integers(0, vocab, size=(G, N, stride)), base).astype(np.int32)
    lens = np.where(rng.random((G, N)) < 0.7, K, rng.integers(0, K + 1, size=(G, N))).astype(np.int32)
    _, _, mean, _ = oracle.gate(seqs, lens, K, 0.1, 0, threads=8)
    s, l = torch.from_numpy(seqs).cuda(), torch.from_numpy(lens).cuda()
    ws = torch.empty(sr.sr_gate_workspace_bytes(G, N, stride, K), dtype=torch.uint8, device="cuda")
    for thr in (float(np.median(mean)), float(np.nextafter(np.quantile(mean, 0.25, method="nearest"), 2.0)), 0.12, 2.0, 0.0):
        stop = torch.full((G,), 9, dtype=torch.uint8, device="cuda")
        sr.sr_gate_decide(s, l, K, thr, 0, stop=stop, workspace=ws)
        assert np.array_equal(stop.cpu().numpy(), (mean < thr).astype(np.uint8)), thr
