"""Logged figures at the sizes where their kernels change shape: one cluster or a whole grid, odd group
sizes, bigrams that fight for slots, rollouts that are equal up to their lengths."""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_05802_b200 as sr

pytestmark = pytest.mark.gpu
dev = torch.device("cuda:0")


@pytest.mark.parametrize("G", [1, 255, 2048, 2049, 8192, 16384, 16385])
@pytest.mark.parametrize("N", [2, 8, 13])
def test_batch_stats(G, N):
    rng = np.random.default_rng(G + N)
    adv = rng.standard_normal((G, N)).astype(np.float32)
    adv[rng.random((G, N)) < 0.3] = 0.0
    stop = (rng.random(G) < 0.4).astype(np.uint8) * 3
    counts = torch.full((3,), -7, dtype=torch.int64, device=dev)
    sumsq = torch.full((2,), -7.0, dtype=torch.float64, device=dev)
    sr.sr_batch_stats(torch.from_numpy(adv).to(dev), torch.from_numpy(stop).to(dev), counts=counts, sumsq=sumsq)
    want = oracle.batch_stats(adv, stop)
    assert np.array_equal(counts.cpu().numpy(), np.asarray(want[0]))
    assert np.allclose(sumsq.cpu().numpy(), np.asarray(want[1]), rtol=1e-12, atol=0)


@pytest.mark.parametrize("G,N,off", [(3000, 32, 0), (8192, 32, 0), (8193, 32, 0), (4096, 32, 1), (4097, 32, 1), (16384, 24, 0), (8456, 31, 0),
                                     (8457, 31, 0), (13107, 20, 1), (13108, 20, 1), (2304, 5, 3)])
def test_batch_stats_where_one_cluster_ends(G, N, off):
    """Either side of the largest batch one cluster takes, with rows on and off 16 bytes."""
    rng = np.random.default_rng(G + N)
    adv = rng.standard_normal((G, N)).astype(np.float32)
    adv[rng.random((G, N)) < 0.3] = 0.0
    stop = (rng.random(G) < 0.4).astype(np.uint8)
    given = torch.empty(G * N + off, device=dev)[off:].view(G, N)
    given.copy_(torch.from_numpy(adv))
    counts = torch.full((3,), -7, dtype=torch.int64, device=dev)
    sumsq = torch.full((2,), -7.0, dtype=torch.float64, device=dev)
    sr.sr_batch_stats(given, torch.from_numpy(stop).to(dev), counts=counts, sumsq=sumsq)
    want = oracle.batch_stats(adv, stop)
    assert np.array_equal(counts.cpu().numpy(), np.asarray(want[0]))
    assert np.allclose(sumsq.cpu().numpy(), np.asarray(want[1]), rtol=1e-12, atol=0)


@pytest.mark.parametrize("n,off", [(8 * 4096, 0), (8 * 4096 + 1, 0), (3 * 4096 - 1, 0), (8 * 4096 + 1, 1), (3 * 4096 - 1, 3), (1000003, 1)])
def test_kept_groups(n, off):
    rng = np.random.default_rng(n)
    stop, zv = ((rng.random(n) < 0.3).astype(np.uint8) for _ in range(2))
    index = torch.full((n,), -7, dtype=torch.int32, device=dev)
    count = torch.full((1,), -7, dtype=torch.int32, device=dev)
    ws = torch.empty(sr.sr_kept_groups_workspace_bytes(n), dtype=torch.uint8, device=dev)
    given = []
    for flags in (stop, zv):                                      # `off` bytes past a 16-byte boundary
        given.append(torch.empty(n + off, dtype=torch.uint8, device=dev)[off:])
        given[-1].copy_(torch.from_numpy(flags))
    sr.sr_kept_groups(*given, index=index, count=count, workspace=ws)
    want = oracle.kept_groups(stop, zv)
    assert int(count) == want.size and np.array_equal(index.cpu().numpy()[:want.size], want)


@pytest.mark.parametrize("N,K", [(2, 0), (2, 32), (3, 5), (4, 17), (7, 31), (9, 1), (16, 2), (19, 30), (32, 32)])
def test_group_signals(N, K):
    rng = np.random.default_rng(100 * N + K)
    G, stride = 61, 36
    seqs = rng.integers(0, rng.choice([2, 9, 1 << 31], size=(G, 1, 1)), size=(G, N, stride)).astype(np.int32)
    seqs[::4] = seqs[::4, :1]                                     # equal but for their lengths
    seqs[1::4, 1::2] = seqs[1::4, :1]
    lens = rng.integers(-1, K + 3, size=(G, N)).astype(np.int32)
    lens[::8] = K
    want = oracle.group_signals(seqs, np.maximum(lens, 0), K)
    outs = [torch.full((G,), -1.0, dtype=torch.float64, device=dev) for _ in range(4)]
    sr.sr_group_signals(torch.from_numpy(seqs).to(dev), torch.from_numpy(lens).to(dev), K, unique_prefix_ratio=outs[0],
                        unique_action_ratio=outs[1], action_entropy=outs[2], bigram_jaccard_mean=outs[3])
    got = [o.cpu().numpy() for o in outs]
    for k in (0, 1, 3):
        assert np.array_equal(got[k].view(np.uint64), want[k].view(np.uint64)), k
    assert np.allclose(got[2], want[2], rtol=0, atol=1e-13)
