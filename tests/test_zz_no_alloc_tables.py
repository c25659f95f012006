"""Allocation-free batched form: instance counts around the number that
travels with the launch (64), and tiles around 1024 streams."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import paper_1609_01257_gb300 as rng

pytestmark = pytest.mark.gpu
U64 = ctypes.c_uint64


@pytest.mark.parametrize("count", [1, 2, 31, 32, 33, 63, 64, 65, 1023, 1025])
def test_instance_tables(count):
    r = np.random.default_rng(count)
    ns = [int(x) for x in r.choice([1, 3, 256, 1023, 1024, 1025, 2048, 2049, 5000], count)]
    ts = [int(x) for x in r.integers(1, 20, count)]
    seeds = [int(x) for x in r.integers(0, 2**63, count)]
    offs, o = [], 0
    for n, t in zip(ns, ts):
        offs.append(o)
        o += n * t + int(r.integers(0, 3))  # some outputs off the 16-byte boundaries
    buf = torch.full((o + 4,), -1, dtype=torch.int64, device="cuda")
    ptrs = (ctypes.c_void_p * count)(*[buf.data_ptr() + 8 * a for a in offs])
    rc = rng.load().rng_batch_generate_noalloc(count, (U64 * count)(*ns), (U64 * count)(*ts), (U64 * count)(*seeds),
                                               ptrs, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), None)
    assert rc == 0
    got = buf.cpu().numpy().view(np.uint64)
    want = np.full(o + 4, 2**64 - 1, dtype=np.uint64)
    for a, n, t, s in zip(offs, ns, ts, seeds):
        want[a:a + n * t] = oracle.generate(n, s, t).reshape(-1)
    assert np.array_equal(got, want)
