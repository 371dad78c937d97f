"""Packed host input of 14 MiB and more, which is gated in two parts on one workspace: groups of several pairs, whose distances begin
elsewhere than the groups do, parts with more pairs than one CTA orders, odd group counts, texts and uniform tokens, one
call after the other on one arena."""
import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches
from paper_2605_05802_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,N,K", [(601, 8, 1024), (1205, 5, 801), (1500, 3, 1000), (301, 16, 1021)])
def test_packed_input_in_two_parts(G, N, K):
    import torch
    import paper_2605_05802_b200 as sr
    rng = np.random.default_rng(G + K)
    stride, P = (K + 3) // 4 * 4, N * (N - 1) // 2
    arena = torch.empty(sr.sr_gate_host_packed_arena_bytes(G, N, stride, K), dtype=torch.uint8, device="cuda:0")
    cs = torch.cuda.Stream()
    batches = []
    for kind in ("tokens", "texts", "few symbols"):
        draw = {"tokens": lambda shape: rng.integers(0, 151936, size=shape), "texts": lambda shape: np.exp(rng.random(shape) * np.log(151936.0)) - 1.0,
                "few symbols": lambda shape: rng.integers(0, 300, size=shape)}[kind]
        rate = rng.choice([0.01, 0.1, 0.5, 1.0], size=(G, 1, 1))
        seqs = np.where(rng.random((G, N, stride)) < rate, draw((G, N, stride)), draw((G, 1, stride))).astype(np.int32)
        lens = rng.integers(K - K // 50, K + 1, size=(G, N)).astype(np.int32)
        lens[G // 2, 0] = lens[G // 2 - 1, N - 1] = 0
        symbols, row_start = W.pack_rows(seqs, lens)
        assert symbols.size * 4 >= 14 << 20
        batches.append((torch.from_numpy(symbols).pin_memory(), torch.from_numpy(row_start).pin_memory(), oracle.gate(seqs, lens, K, 0.3, 0, threads=8)))
    outs = []
    for h_sym, h_rs, _ in batches + batches[:1]:             # (nothing waits in between)
        pd = torch.full((G, P), -7, dtype=torch.int32).pin_memory()
        ps = torch.full((G,), -7, dtype=torch.int32).pin_memory()
        mean = torch.full((G,), -7.0, dtype=torch.float64).pin_memory()
        stop = torch.full((G,), 9, dtype=torch.uint8).pin_memory()
        status = torch.zeros(1, dtype=torch.int32).pin_memory()
        sr.sr_gate_host_packed(h_sym, h_rs, N, stride, K, 0.3, 0, pair_dist=pd, pair_sum=ps, mean=mean, stop=stop, status=status,
                               arena=arena, copy_stream=cs)
        outs.append((pd, ps, mean, stop, status))
    torch.cuda.current_stream().synchronize()
    for (pd, ps, mean, stop, status), (_, _, want) in zip(outs, batches + batches[:1]):
        assert int(status) == 0
        assert_gate_matches((pd.numpy(), ps.numpy(), mean.numpy(), stop.numpy()), want, f"G={G} N={N} K={K}")
