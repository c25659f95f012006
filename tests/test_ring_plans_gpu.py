"""Which kernel a ring takes: the rows of a ring are not split into bands, so
launches of few tiles keep register stores, as do rings on the 128-byte lines
that are small beside the L2; the last rows against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1609_01257_gb300 as rng

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,T,R,kernel", [
    (65_536, 2100, 4, "register"),     # on the lines, 16 tiles
    (70_001, 300, 7, "register"),      # off the lines, 18 tiles
    (311_296, 1030, 2, "register"),    # half as many tiles as SMs
    (1 << 20, 300, 3, "register"),     # on the lines, 24 MB of ring
    (311_297, 40, 3, "bulk"),          # one tile more, off the lines
    (1 << 20, 140, 130, "bulk"),       # on the lines, 1.1 GB of ring
])
def test_kernel_of_a_ring(n, T, R, kernel):
    g = rng.Generator(n, 61)
    ring = torch.zeros((R, n), dtype=torch.int64, device="cuda").view(torch.uint64)
    g.generate_ring(T, ring)
    ran = g.last_launch()["kernel"]
    after = g.generate(1).cpu().numpy()
    g.close()
    last = min(R, 3)
    want = oracle.generate(n, 61, last + 1, p0=T - last)
    got = ring.cpu().numpy()
    for i in range(last):
        assert np.array_equal(got[(T - last + i) % R], want[i]), i
    assert np.array_equal(after[0], want[last])
    assert ran == kernel
