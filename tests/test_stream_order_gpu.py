"""Stream ordering of the generator's calls with torch's current stream: the
tensor handed back is ready for work queued on that stream, whichever it is,
and memory freed by the caller is reused only after the kernel that wrote it."""
import numpy as np
import pytest
import torch

import oracle
import paper_1609_01257_gb300 as rng

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own", [False, True])
def test_results_are_ready_on_the_current_stream(own):
    n, T = 1_000_003, 4
    want = oracle.generate(n, 6, 3 * T)
    s = torch.cuda.Stream()
    g = rng.Generator(n, 6, compute_stream=s if own else None)
    with torch.cuda.stream(s):
        a = g.generate(T).view(torch.int64) + 0   # queued on s right behind the kernel
        b = torch.zeros((T, n), dtype=torch.int64, device="cuda").view(torch.uint64)
        b = g.generate(T, out=b).view(torch.int64) + 0  # after the fill
        for _ in range(3):
            g.generate(1).view(torch.int64).add_(1)  # freed at once, its memory written on s
        x, _sums = g.generate_checksum(T)
    c = torch.stack([a, b]).cpu().numpy() if s.synchronize() is None else None
    g.close()
    assert np.array_equal(c.view(np.uint64).reshape(2 * T, n), want[:2 * T])
    wx, _, _ = oracle.row_checksums(n, 6, T, p0=2 * T + 3)
    assert np.array_equal(x.cpu().numpy(), wx)
