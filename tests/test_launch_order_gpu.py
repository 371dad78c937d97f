"""Calls that follow one another on a stream without synchronisation, each reading what the one
before it wrote: kernels start early (programmatic stream serialisation) but must not read early."""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_05802_b200 as sr
from paper_2605_05802_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("n_groups,K", [(16, 10), (3000, 30), (40, 300)])
def test_back_to_back_calls_see_each_other(n_groups, K, captured):
    dev = torch.device("cuda:0")
    make = (lambda s: W.token_gate(seed=s, n_groups=n_groups, min_len=40, max_len=K)) if K > 32 else \
        (lambda s: W.agent_gate(seed=s, n_groups=n_groups, K=K))
    batches = [make(s) for s in range(4)]
    threshold = 0.4
    host = [(torch.from_numpy(w.seqs).to(dev), torch.from_numpy(w.lens).to(dev), torch.from_numpy(w.rewards).to(dev)) for w in batches]
    seqs, lens, rewards = (torch.empty_like(x) for x in host[0])
    G, N, stride = seqs.shape
    stop, zv = (torch.empty(G, dtype=torch.uint8, device=dev) for _ in range(2))
    adv = torch.empty((G, N), device=dev)
    index, count = torch.zeros(G, dtype=torch.int32, device=dev), torch.zeros(1, dtype=torch.int32, device=dev)
    ws = torch.empty(max(sr.sr_gate_workspace_bytes(G, N, stride, K), 1), dtype=torch.uint8, device=dev)
    kws = torch.empty(sr.sr_kept_groups_workspace_bytes(G), dtype=torch.uint8, device=dev)

    def step():
        sr.sr_gate(seqs, lens, K, threshold, stop=stop, workspace=ws)
        sr.sr_grpo_advantage(rewards, stop, 1e-6, adv=adv, zero_var=zv)
        sr.sr_kept_groups(stop, zv, index=index, count=count, workspace=kws)

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        run = step
        if captured:
            step()
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                step()
            run = graph.replay
        got = []
        for k in range(24):
            for dst, src in zip((seqs, lens, rewards), host[k % 4]):
                dst.copy_(src)
            run()
            got.append([x.clone() for x in (stop, zv, adv, index, count)])
    torch.cuda.synchronize()
    want = []
    for w in batches:
        ostop = oracle.gate(w.seqs, w.lens, K, threshold, threads=8)[3]
        oadv, ozv = oracle.advantage(w.rewards, ostop, 1e-6)
        want.append((ostop, ozv, oadv, oracle.kept_groups(ostop, ozv)))
    for k, (s, z, a, i, c) in enumerate(got):
        ostop, ozv, oadv, oidx = want[k % 4]
        assert np.array_equal(s.cpu().numpy(), ostop) and np.array_equal(z.cpu().numpy(), ozv), k
        assert np.allclose(a.cpu().numpy(), oadv, rtol=1e-6, atol=0), k
        assert int(c) == len(oidx) and np.array_equal(i.cpu().numpy()[:int(c)], oidx), k


@pytest.mark.parametrize("decide", [False, True])
@pytest.mark.parametrize("n_groups,K", [(16, 1024), (16, 512), (5, 200), (300, 1024)])
def test_replayed_multi_word_calls(n_groups, K, decide):
    """The routes of the multi-word gate from one captured graph on changing inputs: the last CTA of a group counts the
    arrivals, a cluster hands over its distances or settles its group from bounds, a sorted batch counts its bins."""
    dev = torch.device("cuda:0")
    batches = [W.token_gate(seed=s, n_groups=n_groups, min_len=40, max_len=K) for s in range(3)]
    host = [(torch.from_numpy(w.seqs).to(dev), torch.from_numpy(w.lens).to(dev)) for w in batches]
    seqs, lens = (torch.empty_like(x) for x in host[0])
    G, N, stride = seqs.shape
    threshold = float(np.median(oracle.gate(batches[0].seqs, batches[0].lens, K, 0.0, threads=8)[2]))
    stop = torch.empty(G, dtype=torch.uint8, device=dev)
    mean = None if decide else torch.empty(G, dtype=torch.float64, device=dev)
    ws = torch.empty(sr.sr_gate_workspace_bytes(G, N, stride, K), dtype=torch.uint8, device=dev)

    def step():
        if decide:
            sr.sr_gate_decide(seqs, lens, K, threshold, stop=stop, workspace=ws)
        else:
            sr.sr_gate(seqs, lens, K, threshold, mean=mean, stop=stop, workspace=ws)

    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        for dst, src in zip((seqs, lens), host[0]):
            dst.copy_(src)
        step()
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            step()
            step()
        got = []
        for k in range(9):
            for dst, src in zip((seqs, lens), host[k % 3]):
                dst.copy_(src)
            graph.replay()
            got.append((stop.clone(), None if decide else mean.clone()))
    torch.cuda.synchronize()
    want = [oracle.gate(w.seqs, w.lens, K, threshold, threads=8) for w in batches]
    for k, (s, m) in enumerate(got):
        assert np.array_equal(s.cpu().numpy(), want[k % 3][3]), k
        assert decide or np.array_equal(m.cpu().numpy(), want[k % 3][2]), k


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("G,N", [(200, 8), (30000, 2), (3571, 8), (12000, 8), (23000, 8), (2173, 24), (70000, 8)])
def test_steps_back_to_back_see_each_other(G, N, captured):
    """Incremental steps without synchronisation between them, at sizes on either side of where a step
    overlaps the one before it."""
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(G + N)
    steps = 9
    actions = np.where(rng.random((steps, G, N)) < 0.6, rng.integers(0, 5, size=(steps, G, 1)), rng.integers(0, 5, size=(steps, G, N))).astype(np.int32)
    given = torch.from_numpy(actions).to(dev)
    state = torch.empty(sr.sr_incr_state_bytes(G, N, steps), dtype=torch.uint8, device=dev)
    mean = torch.empty((steps, G), dtype=torch.float64, device=dev)
    stop = torch.empty((steps, G), dtype=torch.uint8, device=dev)

    def episode():
        sr.sr_incr_init(state, G, N, steps)
        for t in range(steps):
            sr.sr_gate_step_incremental(state, given[t], 0.3, mean=mean[t], stop=stop[t])

    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                episode()
            graph.replay()
        else:
            episode()
    torch.cuda.synchronize()
    mean, stop = mean.cpu().numpy(), stop.cpu().numpy()
    some = np.unique(np.concatenate([rng.integers(0, G, 200), [0, G - 1]]))
    seqs = np.zeros((len(some), N, 12), dtype=np.int32)
    seqs[:, :, :steps] = actions[:, some].transpose(1, 2, 0)
    for t in range(steps):
        want = oracle.gate(seqs, np.full((len(some), N), t + 1, dtype=np.int32), steps, 0.3, threads=8)
        assert np.array_equal(mean[t, some].view(np.uint64), want[2].view(np.uint64)), t
        assert np.array_equal(stop[t, some], want[3]), t
