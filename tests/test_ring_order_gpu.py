"""Rows that come round to the same place of a ring on the bulk-copy kernel:
each copy there waits for the one before it, so that the ring ends with the
last rows.  Ring sizes around the three waits (one row, the row buffers less
two of each shape, 32 rows), many rounds, forced and as the library chooses."""
import numpy as np
import pytest
import torch

import oracle
import paper_1609_01257_gb300 as rng

pytestmark = pytest.mark.gpu


def _check(n, T, R, off=0, **kw):
    g = rng.Generator(n, 47, **kw)
    buf = torch.zeros(R * n + off, dtype=torch.int64, device="cuda")
    ring = buf[off:].view(R, n).view(torch.uint64)
    want = oracle.generate(n, 47, 2 * T)
    for k in range(2):  # from the hash, then from states in memory
        g.generate_ring(T, ring)
        got = ring.cpu().numpy()
        for i in range(max(0, T - R), T):
            assert np.array_equal(got[i % R], want[k * T + i]), (k, i)
    ran = g.last_launch()["kernel"]
    g.close()
    return ran


@pytest.mark.parametrize("R", [1, 2, 4, 5, 6, 7, 10, 11, 12, 31, 32, 33, 200])
@pytest.mark.parametrize("vpt", [4, 8, 16])
def test_forced_bulk_copies(vpt, R):
    assert _check(9001, 173, R, store_policy=2, values_per_thread=vpt) == "bulk"


@pytest.mark.parametrize("R", [1, 2, 5, 12, 32, 33, 100])
@pytest.mark.parametrize("n,T,off", [(70_001, 301, 0), (300_001, 130, 1), (700_001, 70, 0), (622_592, 129, 0)])
def test_as_the_library_chooses(n, T, R, off):
    _check(n, T, R, off)
