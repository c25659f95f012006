"""Which kernel a generate-and-checksum launch takes, and the bit-sliced one
(from 2^27 values and 64 rows) against the CPU oracle: ragged and full tiles of
8192 streams, whole tiles, tiles split by rows over many blocks, row counts off
the 16-row batches, a stream offset, states set by the caller."""
import numpy as np
import pytest
import torch

import oracle
import paper_1609_01257_gb300 as rng

pytestmark = pytest.mark.gpu

TILE = 8192


def _same(got, n, seed, rows, **kw):
    wx, ws, _ = oracle.row_checksums(n, seed, rows, **kw)
    assert np.array_equal(got[0].cpu().numpy(), wx)
    assert np.array_equal(got[1].cpu().numpy(), ws)


@pytest.mark.parametrize("n,rows", [
    (5462, 24_700),          # just over two thirds of one tile, split over every block
    (TILE, 16_400),          # one full tile
    (2 * TILE + 2, 8300),    # a last tile of two streams
    (300_001, 451),          # rows off every batch
    (1 << 21, 64),           # the fewest rows
    (3_735_550, 65),         # whole tiles on three blocks of 152 SMs each
    (3_740_001, 65),         # one tile more: split
    (4_000_037, 67),
])
def test_sliced_checksums_and_continuation(n, rows):
    g = rng.Generator(n, 77)
    for k in range(2):  # from the hash, then from states in memory
        _same(g.generate_checksum(rows), n, 77, rows, p0=k * rows)
        info = g.last_checksum()
        assert info["kernel"] == "sliced"
        if not info["band_rows"]:
            assert info["grid"] == -(-n // TILE)
    tail = g.generate(2).cpu().numpy()
    g.close()
    assert np.array_equal(tail, oracle.generate(n, 77, 2, p0=2 * rows))
    slots = 3 * torch.cuda.get_device_properties(0).multi_processor_count
    if -(-n // TILE) < slots * 0.9:  # an unfilled wave is split
        assert info["band_rows"] > 0
    if -(-n // TILE) == slots:
        assert info["band_rows"] == 0


def test_sliced_checksums_with_offset_and_set_states():
    n, rows, off = 70_000, 1950, 2**32 - 70_000
    g = rng.Generator(n, 5, stream_offset=off)
    g.skip(9)
    _same(g.generate_checksum(rows), n, 5, rows, p0=9, g0=off)
    assert g.last_checksum()["kernel"] == "sliced"
    # arbitrary states, zero among them, against the values themselves
    st = np.random.default_rng(3).integers(0, 2**64, n, dtype=np.uint64)
    st[::1001] = 0
    g.set_state(st, 0)
    x, s = (v.cpu().numpy() for v in g.generate_checksum(rows))
    assert g.last_checksum()["kernel"] == "sliced"
    g.set_state(st, 0)
    values = g.generate(rows).cpu().numpy()
    g.close()
    assert np.array_equal(x, np.bitwise_xor.reduce(values, axis=1))
    assert np.array_equal(s, values.sum(axis=1, dtype=np.uint64))


@pytest.mark.parametrize("n,rows,kw", [
    (1 << 21, 63, {}), (TILE, 16_383, {}), (5461, 24_700, {}), (1 << 21, 64, {"output_mode": 1}),
    (1 << 21, 64, {"values_per_thread": 16}),
])
def test_launches_beside_the_line_take_the_other_kernel(n, rows, kw):
    g = rng.Generator(n, 79, **kw)
    got = g.generate_checksum(rows)
    assert g.last_checksum()["kernel"] == "checksum"
    g.close()
    _same(got, n, 79, rows, output_mode=kw.get("output_mode", 0))


@pytest.mark.parametrize("less,vpt", [(0, 16), (1, 8)])
@pytest.mark.parametrize("mode", [0, 1])
def test_few_rows_of_many_tiles(less, vpt, mode):
    # five tiles of 16 values an SM
    n, rows = 5 * 4096 * torch.cuda.get_device_properties(0).multi_processor_count - less, 15
    g = rng.Generator(n, 81, output_mode=mode)
    got = g.generate_checksum(rows)
    assert g.last_checksum()["values_per_thread"] == vpt
    g.close()
    _same(got, n, 81, rows, output_mode=mode)


def test_no_checksum_launch_yet():
    g = rng.Generator(100, 1)
    with pytest.raises(rng.RngError):
        g.last_checksum()
    g.close()
