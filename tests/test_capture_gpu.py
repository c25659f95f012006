"""Launches captured into a graph and replayed, between eager launches of other
lengths: every replay goes on from the states that the launch before it left,
also where eager launches run in bands (two state arrays, tables per length)."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_1609_01257_gb300 as rng
from paper_1609_01257_gb300 import _capi

pytestmark = pytest.mark.gpu


class _Call:
    """Rows or checksums of T iterations into memory of its own."""

    def __init__(self, g, kind, T, seed, mode):
        self.g, self.kind, self.T, self.seed, self.mode = g, kind, T, seed, mode
        shape = (T, g.streams) if kind == "rows" else (2, T)
        self.out = torch.zeros(shape, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()

    def __call__(self):
        if self.kind == "rows":
            self.g.generate_to(self.T, self.out.data_ptr())
        else:
            p = self.out.data_ptr()
            _capi.check(self.g._lib.rng_generate_checksum, self.g._h, self.T, ctypes.c_void_p(p),
                        ctypes.c_void_p(p + 8 * self.T))

    def right(self, p0):
        torch.cuda.synchronize()
        got = self.out.cpu().numpy().view(np.uint64)
        n = self.g.streams
        if self.kind == "rows":
            return np.array_equal(got, oracle.generate(n, self.seed, self.T, p0=p0, output_mode=self.mode))
        x, s, _ = oracle.row_checksums(n, self.seed, self.T, p0=p0, output_mode=self.mode)
        return np.array_equal(got[0], x) and np.array_equal(got[1], s)


@pytest.mark.parametrize("kind,n,T,T2,mode", [
    ("sum", 1001, 100, 300, 0), ("sum", 65_536, 200, 1000, 0), ("sum", 65_536, 300, 200, 1),
    ("sum", 8192, 17_000, 20_000, 0), ("sum", 300_001, 460, 100, 0), ("sum", 1_300_001, 130, 70, 1),
    ("rows", 1001, 100, 2000, 0), ("rows", 20_001, 200, 300, 1), ("rows", 4096, 9000, 8500, 0),
    ("rows", 65_537, 300, 129, 0),
])
@pytest.mark.parametrize("warm", [False, True])
def test_replays_and_eager_launches_take_turns(kind, n, T, T2, mode, warm):
    seed = 89
    g = rng.Generator(n, seed, profiling=False, output_mode=mode)
    g.skip(1)
    p = 1
    call, other = _Call(g, kind, T, seed, mode), _Call(g, kind, T2, seed, mode)
    if warm:  # an eager launch has taken the memory for bands
        for c in (call, other, call):
            c()
            p += c.T
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=g.stream):
        call()
    # Recorded, not run: the same length eagerly, then another one.
    for c in (call, other):
        c()
        assert c.right(p)
        p += c.T
    for k in range(3):
        graph.replay()
        assert call.right(p), k
        p += T
        c = (other, call)[k % 2]
        c()
        assert c.right(p), k
        p += c.T
    g.close()


@pytest.mark.parametrize("kind,n,T", [("rows", 4096, 20_000), ("rows", 5000, 400), ("sum", 65_536, 300),
                                      ("sum", 8192, 17_000)])
def test_a_captured_run_from_the_start(kind, n, T):
    seed = 97
    g = rng.Generator(n, seed, profiling=False)
    call, more = _Call(g, kind, T, seed, 0), _Call(g, kind, T - 150, seed, 0)
    call()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=g.stream):
        g.init()
        call()
    for _ in range(2):  # every replay starts the streams over
        graph.replay()
        assert call.right(0)
        more()
        assert more.right(T)
    g.close()


def test_a_captured_skip():
    n, T = 70_001, 300
    g = rng.Generator(n, 101, profiling=False)
    call = _Call(g, "rows", T, 101, 0)
    call()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=g.stream):
        g.skip(1000)
    p = T
    for _ in range(2):
        graph.replay()
        p += 1000
        call()
        assert call.right(p)
        p += T
    g.close()
