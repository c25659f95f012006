"""Bit-sliced generate-and-checksum (chosen for output mode 0 from 2^25 values
and 64 rows up) against the CPU oracle: ragged and full tiles of 8192 streams,
tiles split by rows (from the hash, and from states in memory, where the final
states go to a second array), row counts off the 16-row batches, offsets,
states set by the caller, and the streams' continuation after it."""
import numpy as np
import pytest

import oracle
import paper_1609_01257_gb300 as rng

pytestmark = pytest.mark.gpu


def _same(got, n, seed, rows, **kw):
    wx, ws, _ = oracle.row_checksums(n, seed, rows, **kw)
    assert np.array_equal(got[0].cpu().numpy(), wx)
    assert np.array_equal(got[1].cpu().numpy(), ws)


@pytest.mark.parametrize("n,rows", [
    (5462, 6200),        # just over two thirds of one tile, split over every block
    (8192, 4099),        # one full tile
    (8193 * 2, 2051),    # a last tile of two streams
    (300_001, 113),      # rows off every batch
    (524_288, 64),       # the fewest rows
    (3_740_001, 65),     # just under one wave of whole tiles
    (4_000_037, 67),     # a second wave: split
])
def test_sliced_checksums_and_continuation(n, rows):
    g = rng.Generator(n, 77)
    _same(g.generate_checksum(rows), n, 77, rows)             # from the hash
    _same(g.generate_checksum(rows), n, 77, rows, p0=rows)    # from states in memory
    tail = g.generate(2).cpu().numpy()
    g.close()
    assert np.array_equal(tail, oracle.generate(n, 77, 2, p0=2 * rows))


def test_sliced_checksums_with_offset_and_set_states():
    n, rows, off = 70_000, 501, 2**32 - 70_000
    g = rng.Generator(n, 5, stream_offset=off)
    g.skip(9)
    _same(g.generate_checksum(rows), n, 5, rows, p0=9, g0=off)
    # arbitrary states, zero among them: checked against the same states
    # taken through the values themselves
    st = np.random.default_rng(3).integers(0, 2**64, n, dtype=np.uint64)
    st[::1001] = 0
    g.set_state(st, 0)
    x, s = (v.cpu().numpy() for v in g.generate_checksum(rows))
    g.set_state(st, 0)
    rows_out = g.generate(rows).cpu().numpy()
    g.close()
    assert np.array_equal(x, np.bitwise_xor.reduce(rows_out, axis=1))
    assert np.array_equal(s, rows_out.sum(axis=1, dtype=np.uint64))
