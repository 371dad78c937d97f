"""Single-word gate through the kernel that names symbols: batches large enough to leave the direct
comparison, two patterns per word up to K = 15, a warp or a CTA per group above, odd group sizes,
lengths around quads, symbols that occur once, everywhere, or fight for one slot of the table."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from helpers import assert_gate_matches, gate_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,pairs", [(8, 15, 40000), (8, 9, 100000), (9, 12, 100000), (11, 14, 40000), (16, 13, 40000), (32, 3, 300000),
                                       (31, 15, 120000), (32, 15, 120000), (17, 1, 300000), (12, 7, 1000000), (31, 11, 1200000),
                                       (8, 16, 25000), (14, 16, 25000), (2, 17, 37), (3, 32, 111), (5, 31, 370), (8, 32, 1036),
                                       (8, 17, 1036), (9, 16, 25000), (9, 17, 1332), (13, 29, 2886), (32, 32, 18352), (31, 18, 17205)])
@pytest.mark.parametrize("symbols", ["few", "base", "wide", "crowd"])
def test_named_gate(N, K, pairs, symbols):
    P = N * (N - 1) // 2
    G = pairs // P + 3                       # up to K = 16: just enough pairs for this kernel
    rng = np.random.default_rng(1000 * N + K)
    stride = (K + 3) // 4 * 4 + 4
    if symbols == "few":
        seqs = rng.integers(0, 5, size=(G, N, stride))
    elif symbols == "base":
        base = rng.integers(0, 4096, size=(G, 1, stride))
        seqs = np.where(rng.random((G, N, stride)) < rng.beta(0.5, 2.0, size=(G, 1, 1)),
                        rng.integers(0, 4096, size=(G, N, stride)), base)
    elif symbols == "wide":
        seqs = rng.integers(-2 ** 31, 2 ** 31, size=(G, N, stride))
    else:                                    # one home slot under the first hash
        inverse = pow(0x9E3779B1, -1, 1 << 32)
        crowd = (((3 << 24) + np.arange(64, dtype=np.uint64)) * np.uint64(inverse) % np.uint64(1 << 32)).astype(np.uint32).view(np.int32)
        seqs = rng.choice(crowd, size=(G, N, stride))
    lens = rng.integers(0, K + 3, size=(G, N)).astype(np.int32)
    lens[::3] = K
    lens[1::7, 0] = -1
    seqs = seqs.astype(np.int32)
    want = oracle.gate(seqs, np.maximum(lens, 0), K, 0.3, threads=8)
    assert_gate_matches(gate_gpu(seqs, lens, K, 0.3), want, f"N={N} K={K} {symbols}")


_THREADS = """
import sys, threading
sys.path[:0] = [{root!r}, {root!r} + "/tests"]
import numpy as np
import oracle
from helpers import assert_gate_matches, gate_gpu
rng = np.random.default_rng(5)
gate_gpu(rng.integers(0, 9, size=(2, 4, 8)).astype(np.int32), None, 8, 0.3)      # set-up, one thread
shapes = [(32, 32), (27, 28), (29, 32), (25, 32), (32, 25), (30, 30), (28, 32), (26, 32)]
inputs = [rng.integers(0, 40, size=(5, N, 32)).astype(np.int32) for N, K in shapes]
outs, gate = [None] * len(shapes), threading.Barrier(len(shapes))
def work(k):
    gate.wait()
    for _ in range(3): outs[k] = gate_gpu(inputs[k], None, shapes[k][1], 0.3)
threads = [threading.Thread(target=work, args=(k,)) for k in range(len(shapes))]
[t.start() for t in threads]; [t.join() for t in threads]
for (N, K), seqs, got in zip(shapes, inputs, outs):
    assert got is not None, (N, K)
    assert_gate_matches(got, oracle.gate(seqs, None, K, 0.3), (N, K))
print("threads ok")
"""


def test_first_large_calls_of_several_threads():
    """Shapes that need more than 48 KB of shared memory, called for the first time in a process by
    several threads at once: none may be refused for what another one has asked for."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", _THREADS.format(root=root)], capture_output=True, text=True, timeout=600)
    assert out.returncode == 0 and "threads ok" in out.stdout, out.stdout + out.stderr
