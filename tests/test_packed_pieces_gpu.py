"""Packed host input on either side of the size from which it is sent in pieces: equal to the oracle, one call after
the other on one arena, with rows without symbols and group counts that the pieces do not divide; the last one is gated in two parts."""
import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches
from paper_2605_05802_b200 import workloads as W


@pytest.mark.gpu
@pytest.mark.parametrize("G,N,K", [(64, 8, 1000), (66, 8, 1024), (67, 16, 520), (131, 5, 1001), (1901, 2, 1024)])
def test_packed_input_in_pieces(G, N, K):
    import torch
    import paper_2605_05802_b200 as sr
    w = W.token_gate(seed=G + K, n_groups=G, min_len=K - 8, max_len=K, N=N, vocab=3000)
    lens = w.lens.copy()
    lens[G // 2, 0] = lens[G - 1, N - 1] = 0
    stride, P = w.seqs.shape[2], N * (N - 1) // 2
    want = oracle.gate(w.seqs, lens, K, 0.3, 0, threads=8)
    symbols, row_start = W.pack_rows(w.seqs, lens)
    h_sym, h_rs = torch.from_numpy(symbols).pin_memory(), torch.from_numpy(row_start).pin_memory()
    arena = torch.empty(sr.sr_gate_host_packed_arena_bytes(G, N, stride, K), dtype=torch.uint8, device="cuda:0")
    cs = torch.cuda.Stream()
    for _ in range(3):
        pd = torch.full((G, P), -7, dtype=torch.int32).pin_memory()
        ps = torch.full((G,), -7, dtype=torch.int32).pin_memory()
        mean = torch.full((G,), -7.0, dtype=torch.float64).pin_memory()
        stop = torch.full((G,), 9, dtype=torch.uint8).pin_memory()
        sr.sr_gate_host_packed(h_sym, h_rs, N, stride, K, 0.3, 0, pair_dist=pd, pair_sum=ps, mean=mean, stop=stop,
                               arena=arena, copy_stream=cs)
        torch.cuda.current_stream().synchronize()
        assert_gate_matches((pd.numpy(), ps.numpy(), mean.numpy(), stop.numpy()), want, f"G={G} N={N} K={K}")
