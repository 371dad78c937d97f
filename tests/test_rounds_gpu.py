"""Batches whose tasks outnumber the warps of the recurrence: rounds of tasks that take as long each, whose last one is shared
out evenly, and tasks of many lengths, which are pulled one by one."""
import statistics

import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches, gate_gpu

pytestmark = pytest.mark.gpu


# Tasks on 148 SMs, in the order of the cases: 3750 and 6376 that take as long each, run by sixteen warps an SM, 2433 and 5128 by
# twelve; 2933 of many lengths by twelve, 5789 by sixteen.  (The recurrence has 2368 warps of sixteen, 1776 of twelve.)
@pytest.mark.parametrize("N,K,G,ragged", [(4, 64, 20000, False), (4, 64, 34000, False), (8, 256, 1390, False), (8, 256, 2930, False),
                                          (5, 130, 9000, True), (5, 130, 18000, True)])
def test_every_task_is_run_once(N, K, G, ragged):
    rng = np.random.default_rng(K + G)
    unique, stride = 120, (K + 3) // 4 * 4
    base = rng.integers(0, 10 ** 5, size=(unique, 1, 2 * stride), dtype=np.int32)
    base[:, :, ::5] = rng.integers(0, 12, size=base[:, :, ::5].shape)                 # symbols with mask rows
    move = rng.choice(3, size=(unique, N, stride), p=[0.06, 0.88, 0.06])              # inserted and deleted symbols
    at = np.cumsum(move, axis=2) - move
    some = np.take_along_axis(np.broadcast_to(base, (unique, N, 2 * stride)), at, axis=2)
    some = np.where(move == 0, rng.integers(0, 10 ** 5, size=some.shape), some).astype(np.int32)
    some_lens = rng.integers(K // 8, K + 1, size=(unique, N)).astype(np.int32) if ragged else np.full((unique, N), K, dtype=np.int32)
    which = rng.integers(0, unique, size=G)
    want = oracle.gate(some, some_lens, K, 0.12, threads=8)
    assert_gate_matches(gate_gpu(some[which], some_lens[which], K, 0.12), tuple(x[which] for x in want), f"G={G} N={N} K={K}")


def test_last_round_is_shared_out():
    """2802 tasks that take as long each take 1.6 times what 1772 do on twelve warps an SM, 1.8 where schedulers that ask first
    have three more of them and others none."""
    import torch
    import paper_2605_05802_b200 as sr
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the batches' tasks are counted for 148 SMs")
    N, K = 8, 1024
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    times = []
    for G in (253, 400):
        base = torch.randint(0, 151936, (G, 1, 2 * K), generator=gen, device="cuda", dtype=torch.int32)
        own = torch.randint(0, 151936, (G, N, K), generator=gen, device="cuda", dtype=torch.int32)
        hit = torch.rand((G, N, K), generator=gen, device="cuda") < 0.05
        op = torch.randint(0, 3, (G, N, K), generator=gen, device="cuda")
        move = torch.where(hit & (op == 1), 0, torch.where(hit & (op == 2), 2, 1))
        at = torch.cumsum(move, 2) - move + (hit & (op == 2)).long()
        seqs = torch.where(hit & (op < 2), own, torch.gather(base.expand(G, N, 2 * K), 2, at)).contiguous()
        mean, stop = torch.empty(G, dtype=torch.float64, device="cuda"), torch.empty(G, dtype=torch.uint8, device="cuda")
        ws = torch.empty(sr.sr_gate_workspace_bytes(G, N, K, K), dtype=torch.uint8, device="cuda")
        taken = []
        for _ in range(9):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(5):
                sr.sr_gate(seqs, None, K, 0.12, mean=mean, stop=stop, workspace=ws)
            b.record()
            b.synchronize()
            taken.append(a.elapsed_time(b))
        times.append(statistics.median(taken))
    assert times[1] <= 1.72 * times[0], times
