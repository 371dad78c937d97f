"""sr_gate_decide with nothing but the mask wanted, where groups may be settled from their upper bounds as well: equal to
the oracle at thresholds among the batch's own d_K values and just beside them, in batches whose groups have a cluster each
and in batches that are sorted into warp tasks."""
import numpy as np
import pytest

import oracle


@pytest.mark.gpu
@pytest.mark.parametrize("G,N,K,vocab", [(40, 8, 300, 40), (25, 5, 520, 2000), (30, 2, 70, 9), (12, 16, 200, 60), (70, 11, 90, 300), (300, 8, 260, 500), (62, 8, 1000, 3000), (900, 2, 600, 300)])
def test_mask_alone(G, N, K, vocab):
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
