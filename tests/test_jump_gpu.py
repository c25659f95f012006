"""Jump-ahead kernels at the sizes where they change: the nine-lookup kernel
(from 3 x 2^20 streams) with full and ragged strides, from the hash and from
states in memory, and the table kernel of banded launches with many bands."""
import numpy as np
import pytest

import oracle
import paper_1609_01257_gb300 as rng

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(3 << 20) - 1, 3 << 20, (3 << 20) + 1, 152 * 1024 * 4 * 7 + 777])
def test_wide_jump_from_hash_and_states(n):
    g = rng.Generator(n, 19)
    g.skip(37)
    a = g.generate(1).cpu().numpy()       # position 38: the states are in memory
    g.skip(5)
    b = g.generate(1).cpu().numpy()       # position 44
    g.skip((1 << 64) - 1 - 44)            # the rest of the period
    c = g.generate(1).cpu().numpy()
    g.close()
    for got, p in ((a, 37), (b, 43), (c, 0)):
        assert np.array_equal(got, oracle.generate(n, 19, 1, p0=p)), p


@pytest.mark.parametrize("n,T", [(64, 140_000), (300, 70_003), (5000, 4096)])
def test_many_bands(n, T):
    g = rng.Generator(n, 23)
    a = g.generate(T).cpu().numpy()
    assert g.last_launch()["band_rows"] > 0
    b = g.generate(2).cpu().numpy()
    g.close()
    want = oracle.generate(n, 23, T + 2)
    assert np.array_equal(a, want[:T]) and np.array_equal(b, want[T:])
