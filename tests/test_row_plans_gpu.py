"""Row launches at the edges of the library's own plans (values per thread and
shape left to it) against the CPU oracle: several rows per bulk copy up to 4096
streams, one wide tile up to 6144, balanced tiles and bands above, register
stores for small launches off the lines; outputs off the 16-byte boundaries
with canaries, the stronger output, continuation from the states a banded
launch left, rings, and capture into a graph."""
import numpy as np
import pytest
import torch

import oracle
import paper_1609_01257_gb300 as rng

pytestmark = pytest.mark.gpu


def _check(n, T, off=0, mode=0, kernel=None):
    buf = torch.full((T * n + off + 8,), -1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()  # generate_to launches on the library's stream
    g = rng.Generator(n, 29, output_mode=mode)
    g.generate_to(T, buf.data_ptr() + 8 * off)
    ran = g.last_launch()["kernel"]
    b = g.generate(3).cpu().numpy()   # from the states the launch left
    c = g.generate(T).cpu().numpy()   # the same plan from states in memory
    g.close()
    got = buf.cpu().numpy().view(np.uint64)
    want = oracle.generate(n, 29, 2 * T + 3, output_mode=mode)
    assert np.array_equal(got[off:off + T * n].reshape(T, n), want[:T])
    assert (got[:off] == np.uint64(2**64 - 1)).all() and (got[off + T * n:] == np.uint64(2**64 - 1)).all()
    assert np.array_equal(b, want[T:T + 3]) and np.array_equal(c, want[T + 3:])
    assert kernel is None or ran == kernel, ran


@pytest.mark.parametrize("n", [1, 3, 31, 255, 257, 511, 513, 1023, 1025, 2047, 2049, 4095])
@pytest.mark.parametrize("T,off", [(64, 0), (77, 1), (2500, 3)])
def test_several_rows_per_copy(n, T, off):
    _check(n, T, off, kernel="bulk")


@pytest.mark.parametrize("n,T", [(16, 2432), (256, 4001), (512, 2500), (1024, 2500), (4096, 8192)])
def test_several_rows_per_copy_on_the_lines(n, T):
    _check(n, T, kernel="bulk")


@pytest.mark.parametrize("n,T,off", [(4097, 128, 0), (6143, 301, 1), (6144, 130, 1), (6145, 128, 0), (8193, 200, 5),
                                     (65_537, 129, 0), (131_073, 140, 1), (155_649, 40, 0), (311_297, 33, 1),
                                     (622_593, 32, 0), (622_609, 35, 1)])
def test_wide_and_balanced_tiles(n, T, off):
    _check(n, T, off, kernel="bulk")


@pytest.mark.parametrize("n,T", [(4097, 127), (30_001, 5), (65_537, 63), (102_401, 100), (155_647, 31), (393_215, 9)])
def test_register_stores_for_small_launches_off_the_lines(n, T):
    _check(n, T, 1, kernel="register")


@pytest.mark.parametrize("n,T", [(257, 300), (5001, 130), (70_001, 128), (700_001, 33)])
def test_stronger_output(n, T):
    _check(n, T, 1, mode=1)


@pytest.mark.parametrize("n,T,R", [(1001, 100, 7), (70_001, 140, 3), (700_001, 40, 17)])
def test_rings(n, T, R):
    g = rng.Generator(n, 21)
    ring = torch.zeros((R, n), dtype=torch.int64, device="cuda").view(torch.uint64)
    g.generate_ring(T, ring)
    got = ring.cpu().numpy()
    after = g.generate(1).cpu().numpy()
    g.close()
    want = oracle.generate(n, 21, T + 1)
    for i in range(T - R, T):
        assert np.array_equal(got[i % R], want[i]), i
    assert np.array_equal(after[0], want[T])


@pytest.mark.parametrize("n,T", [(1001, 100), (20_001, 200), (131_073, 300)])
def test_captured_launches_advance_on_replay(n, T):
    # Shapes that run in bands outside a capture: a replay goes on from the
    # states the last one left.
    g = rng.Generator(n, 3, profiling=False)
    g.skip(1)
    out = torch.zeros((T, n), dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=g.stream):
        g.generate_to(T, out.data_ptr())
    want = oracle.generate(n, 3, 2 * T + 1)
    for k in range(2):
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().view(np.uint64), want[1 + k * T:1 + (k + 1) * T]), k
    g.close()
