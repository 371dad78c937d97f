"""The packed tests on match streams, compiled for the host, against their definition entry by entry."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_05802_b200", "csrc")
NONE, ROW, CHAIN = 0x7FFF, 0x8000, 0xC000


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("words")
    src, out = d / "words.cpp", d / "words.so"
    src.write_text('#include "stream_words.cuh"\n'
                   'extern "C" void beside(const uint32_t* v, const uint32_t* at, int n, int strip, uint32_t* out)\n'
                   '{ for (int k = 0; k < n; ++k) out[k] = sr::matches_beside(v[k], at[k], strip); }\n')
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-o", str(out), str(src)])
    return ctypes.CDLL(str(out))


@pytest.mark.parametrize("strip", [0, 4, 32, 300, 992, 1023])
def test_matches_beside(lib, strip):
    """Every node of a pair has its place at or behind the removed prefix: no other one is looked up."""
    rng = np.random.default_rng(strip)
    near = np.clip([strip - 129, strip - 128, strip - 1, strip, strip + 1], 0, 1026)
    edges = np.concatenate([near, [0, 1, 1023, 1026, NONE, ROW, ROW + 1, ROW + 127, CHAIN, CHAIN + strip, CHAIN + 1023]])
    low, high = np.meshgrid(edges, edges)
    entry = np.stack([low.ravel(), high.ravel()], 1).astype(np.uint32)
    column = np.full(entry.shape, strip, np.uint32)
    column[:, 1] += 1
    same = rng.random(entry.shape) < 0.3                     # a match on the main diagonal itself
    entry = np.where(same, column, entry)
    v, at = entry[:, 0] | entry[:, 1] << 16, column[:, 0] | column[:, 1] << 16
    got = np.zeros_like(v)
    lib.beside(v.ctypes.data_as(ctypes.c_void_p), at.ctypes.data_as(ctypes.c_void_p), len(v), strip, got.ctypes.data_as(ctypes.c_void_p))
    want = (entry != NONE) & (entry != column) & ((entry >= strip) | (entry >= ROW))
    assert np.array_equal(got, np.where(want[:, 0], 0x8000, 0) | np.where(want[:, 1], 0x80000000, 0))
