"""Rules of the library's own plans for device rows, on both sides of each line:
kernel and values per thread of the launch, and all values against the oracle,
from the hash and then from states in memory."""
import numpy as np
import pytest
import torch

import oracle
import paper_1609_01257_gb300 as rng

pytestmark = pytest.mark.gpu


def _check(n, T, off, kernel, vpt, mode=0):
    buf = torch.full((T * n + off,), -1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()  # generate_to launches on the library's stream
    g = rng.Generator(n, 71, output_mode=mode)
    want = oracle.generate(n, 71, 2 * T, output_mode=mode)
    for k in range(2):
        g.generate_to(T, buf.data_ptr() + 8 * off)
        g.sync()
        got = buf.cpu().numpy().view(np.uint64)[off:].reshape(T, n)
        assert np.array_equal(got, want[k * T:(k + 1) * T]), k
    info = g.last_launch()
    g.close()
    assert (info["kernel"], info["values_per_thread"]) == (kernel, vpt)


@pytest.mark.parametrize("n,T,off,kernel,vpt", [
    (1 << 21, 16, 1, "bulk", 8),         # off the lines from 2^21 streams: bulk copies from 16 rows
    (1 << 21, 31, 1, "bulk", 8),
    (1 << 21, 15, 1, "staged", 1),
    ((1 << 21) - 1, 31, 0, "staged", 2),
])
def test_few_rows_off_the_lines(n, T, off, kernel, vpt):
    _check(n, T, off, kernel, vpt)


@pytest.mark.parametrize("n,T,kernel,vpt", [(4096, 64, "register", 1), (4096, 127, "register", 1),
                                            (4096, 128, "bulk", 16), (1040, 127, "register", 1),
                                            (1024, 64, "bulk", 4)])
def test_few_streams_off_a_line(n, T, kernel, vpt):
    _check(n, T, 1, kernel, vpt)


@pytest.mark.parametrize("n,T,off,vpt", [
    (311_297, 33, 0, 10),    # one tile a block
    (389_120, 33, 1, 10),    # 2560 streams a tile: every value of a thread used
    (389_121, 33, 0, 16),
    (622_593, 40, 0, 10),    # two tiles a block
    (778_240, 33, 1, 10),
    (778_241, 33, 0, 16),
    (1 << 20, 129, 0, 16),   # on the lines
    (720_896, 129, 0, 10),
])
@pytest.mark.parametrize("mode", [0, 1])
def test_shares_of_at_most_ten_values(n, T, off, vpt, mode):
    _check(n, T, off, "bulk", vpt, mode)


@pytest.mark.parametrize("R", [1, 7, 8, 9, 32, 33])
def test_rings_with_ten_values(R):
    n, T = 330_001, 70
    g = rng.Generator(n, 73)
    ring = torch.zeros((R, n), dtype=torch.int64, device="cuda").view(torch.uint64)
    g.generate_ring(T, ring)
    got = ring.cpu().numpy()
    info = g.last_launch()
    g.close()
    want = oracle.generate(n, 73, T)
    assert (info["kernel"], info["values_per_thread"]) == ("bulk", 10)
    for i in range(T - R, T):
        assert np.array_equal(got[i % R], want[i]), i
