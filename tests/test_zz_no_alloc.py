"""sr_gate_noalloc: the gate for callers that are not allowed to allocate device
memory (a rollout worker living inside an inference engine or trainer that has
already claimed the GPU's memory).  Its scratch is a fixed array inside the
library, so this file checks that it (a) refuses problems that do not fit, on the
host, and (b) gives exactly sr_gate's results, call after call, although every call
reuses the same array with the previous call's leftovers in it.

Collected last on purpose: a run that stops at the first failure has then already
run every other test."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle

import paper_2605_05802_b200 as sr
from paper_2605_05802_b200 import binding, build, workloads as W


def test_noalloc_refuses_what_does_not_fit_before_touching_the_gpu():
    build.build()
    lib = binding.load()
    limit = lib.sr_gate_noalloc_limit_bytes()
    assert limit == 16 << 20
    fake = 1 << 20                       # never dereferenced: the call is refused on the host
    assert lib.sr_gate_workspace_bytes(1024, 8, 1024, 1024) > limit
    rc = lib.sr_gate_noalloc(fake, None, 1024, 8, 1024, 1024, 0.12, 0, None, None, None, fake, None, None)
    assert rc == binding.SR_ERR_SCRATCH_LIMIT
    assert b"scratch" in lib.sr_strerror(rc)
    assert lib.sr_gate_noalloc(fake, None, 4, 1, 64, 64, 0.12, 0, None, None, None, fake, None, None) == binding.SR_ERR_BAD_N
    assert lib.sr_gate_noalloc(fake, None, 4, 8, 64, 65, 0.12, 0, None, None, None, fake, None, None) == binding.SR_ERR_BAD_K
    # an invalid call reports its own error even when the problem would not fit either
    assert lib.sr_gate_noalloc(fake, None, 1024, 8, 1024, 1024, 0.12, 7, None, None, None, fake, None, None) == binding.SR_ERR_BAD_MODE
    assert lib.sr_gate_noalloc(None, None, 1024, 8, 1024, 1024, 0.12, 0, None, None, None, fake, None, None) == binding.SR_ERR_NULL
    assert lib.sr_gate_noalloc(fake + 4, None, 1024, 8, 1024, 1024, 0.12, 0, None, None, None, fake, None, None) == binding.SR_ERR_ALIGN


def _run(fn, w, thr, **extra):
    dev = torch.device("cuda:0")
    G, N, stride = w.seqs.shape
    P = N * (N - 1) // 2
    seqs = torch.from_numpy(w.seqs).to(dev)
    lens = torch.from_numpy(w.lens).to(dev)
    pd = torch.full((G, P), -1, dtype=torch.int32, device=dev)
    ps = torch.full((G,), -1, dtype=torch.int32, device=dev)
    mean = torch.full((G,), -1.0, dtype=torch.float64, device=dev)
    stop = torch.full((G,), 7, dtype=torch.uint8, device=dev)
    fn(seqs, lens, w.K, thr, w.norm_mode, pair_dist=pd, pair_sum=ps, mean=mean, stop=stop, **extra)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in (pd, ps, mean, stop)]


@pytest.mark.gpu
def test_noalloc_matches_sr_gate_on_consecutive_calls():
    dev = torch.device("cuda:0")
    # two different multi-word problems back to back, then the first again: the shared
    # array still holds the other problem's match streams and counters each time
    big = W.token_gate(seed=11, n_groups=48, min_len=200, max_len=1024)
    small = W.token_gate(seed=12, n_groups=9, min_len=33, max_len=150, N=5)
    assert sr.sr_gate_workspace_bytes(48, 8, 1024, 1024) <= sr.sr_gate_noalloc_limit_bytes()
    for w in (big, small, big, big):
        G, N, stride = w.seqs.shape
        ws = torch.empty(sr.sr_gate_workspace_bytes(G, N, stride, w.K), dtype=torch.uint8, device=dev)
        want = _run(sr.sr_gate, w, 0.5, workspace=ws)
        got = _run(sr.sr_gate_noalloc, w, 0.5)
        for a, b in zip(got, want):                 # integers and the fp64 d_K bit for bit
            assert a.dtype == b.dtype and np.array_equal(a.view(np.uint8), b.view(np.uint8))
        for a, b in zip(got, oracle.gate(w.seqs, w.lens, w.K, 0.5, w.norm_mode)):   # and the definition itself
            assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
        assert 0 < want[3].sum() < G
    # the single-word path needs no scratch and is served as well
    w1 = W.agent_gate(K=15)
    for a, b in zip(_run(sr.sr_gate_noalloc, w1, 0.5), _run(sr.sr_gate, w1, 0.5)):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))


_LIMITS = """
import sys
sys.path.insert(0, {root!r})
from paper_2605_05802_b200 import binding
lib = binding.load()
up = lambda x: -(-x // 256) * 256
def demand(G, N, K):                       # as sr_gate.h states it
    P, k = N * (N - 1) // 2, -(-K // 8) * 8
    return 16640 + up(G) + 2 * up(4 * G * P) + up(16 * G * P) + up(2 * k * G * N) + up(2 * k * G * P)
largest = dict()
for N in (2, 3, 4, 8, 16, 31, 32):
    for K in (33, 64, 500, 1024):
        G = 1
        while demand(2 * G, N, K) <= 16 << 20: G *= 2
        step = G
        while step:
            if demand(G + step, N, K) <= 16 << 20: G += step
            step //= 2
        largest[N, K] = G
        call = lambda G: lib.sr_gate_noalloc(1 << 20, None, G, N, 1024, K, 0.12, 0, None, None, None, 1 << 20, None, None)
        # no device here: a batch that passes the checks fails at its first CUDA call
        assert call(G) == binding.SR_ERR_CUDA, (G, N, K)
        assert call(G + 1) == binding.SR_ERR_SCRATCH_LIMIT, (G, N, K)
assert (largest[8, 1024], largest[4, 1024], largest[2, 1024], largest[8, 64]) == (225, 812, 2716, 3173), largest
print("limits ok")
"""


def test_noalloc_takes_every_batch_up_to_its_limit():
    """The limit is a formula of its own: it does not move with the gate's workspace."""
    build.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", _LIMITS.format(root=root)], capture_output=True, text=True, timeout=600,
                         env={**os.environ, "CUDA_VISIBLE_DEVICES": ""})
    assert out.returncode == 0 and "limits ok" in out.stdout, out.stdout + out.stderr


@pytest.mark.gpu
@pytest.mark.parametrize("G,N,K", [(142, 8, 1024), (225, 8, 1024), (81, 8, 1023), (2716, 2, 1024), (812, 4, 1024), (877, 8, 256)])
@pytest.mark.parametrize("tokens", ["uniform", "text", "many repeats"])
def test_noalloc_in_parts_and_with_fewer_mask_rows(G, N, K, tokens):
    """Batches near the limit: more than one part, patterns with fewer mask rows than symbols
    that ask for one ("many repeats": 60 symbols, a dozen or more occurrences each)."""
    rng = np.random.default_rng(G + len(tokens))
    stride = (K + 3) // 4 * 4
    if tokens == "uniform":
        draw = lambda *shape: rng.integers(0, 150000, size=shape)
    elif tokens == "text":
        draw = lambda *shape: np.exp(rng.random(shape) * np.log(150000)) - 1
    else:
        draw = lambda *shape: rng.integers(0, 60, size=shape)
    seqs = draw(G, N, stride).astype(np.int32)
    alike = rng.random((G, 1, 1)) < 0.5
    seqs = np.where(alike & (rng.random((G, N, stride)) < 0.9), seqs[:, :1], seqs)
    lens = rng.integers(K // 2, K + 1, size=(G, N)).astype(np.int32)
    lens[::5] = K
    w = W.token_gate(seed=1, n_groups=2, min_len=40, max_len=64)       # for the fields `_run` reads
    w.seqs, w.lens, w.K = np.ascontiguousarray(seqs), lens, K
    ws = torch.empty(sr.sr_gate_workspace_bytes(G, N, stride, K), dtype=torch.uint8, device="cuda:0")
    got, want = _run(sr.sr_gate_noalloc, w, 0.3), _run(sr.sr_gate, w, 0.3, workspace=ws)
    for a, b in zip(got, want):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
    some = np.unique(np.concatenate([rng.integers(0, G, 6), [0, G // 2, G - 1]]))
    for a, b in zip(got, oracle.gate(seqs[some], lens[some], K, 0.3, w.norm_mode, threads=8)):
        assert np.array_equal(a[some].view(np.uint8), b.view(np.uint8))


_FIRST_CALL = """
import sys
sys.path.insert(0, {root!r})
import numpy as np, torch
import oracle
import paper_2605_05802_b200 as sr
from paper_2605_05802_b200 import workloads as W
w = W.token_gate(seed=21, n_groups=6, min_len=40, max_len=260, N=4)
dev = torch.device("cuda:0")
seqs, lens = torch.from_numpy(w.seqs).to(dev), torch.from_numpy(w.lens).to(dev)
G, N, stride = w.seqs.shape
pd = torch.empty((G, N * (N - 1) // 2), dtype=torch.int32, device=dev)
stop = torch.empty(G, dtype=torch.uint8, device=dev)
mean = torch.empty(G, dtype=torch.float64, device=dev)
# the very first library call of this process is the entry point under test
sr.sr_gate_noalloc(seqs, lens, w.K, 0.5, w.norm_mode, pair_dist=pd, mean=mean, stop=stop)
torch.cuda.synchronize()
opd, _, omean, ostop = oracle.gate(w.seqs, w.lens, w.K, 0.5, w.norm_mode)
assert np.array_equal(pd.cpu().numpy(), opd)
assert np.array_equal(mean.cpu().numpy().view(np.uint64), omean.view(np.uint64))
assert np.array_equal(stop.cpu().numpy(), ostop)
print("first-call ok")
"""


@pytest.mark.gpu
def test_first_call_of_a_fresh_process_sets_the_scratch_up():
    """The documented set-up happens inside the first call on a device: check it in a
    process that has made no other library call before."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", _FIRST_CALL.format(root=root)], capture_output=True,
                         text=True, timeout=600)
    assert out.returncode == 0 and "first-call ok" in out.stdout, out.stdout + out.stderr
