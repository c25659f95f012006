"""bench.py's ALU figure of a checksum run: only for runs of the captured kernel
and size, since fewer rows or the other kernel run more operations per value."""
import pytest

import bench


@pytest.mark.parametrize("mode,kernel,streams,rows,ops", [
    (0, "sliced", 1 << 22, 1024, 5.95), (0, "sliced", 1 << 24, 512, 5.95), (0, "sliced", 1 << 22, 511, None),
    (0, "sliced", 8192, 1 << 17, None), (0, "checksum", 1 << 22, 1024, None),
    (1, "checksum", 1 << 22, 64, 9.43), (1, "checksum", 1 << 22, 63, None), (1, "checksum", 65_536, 4096, None),
])
def test_alu_operations_per_value(mode, kernel, streams, rows, ops):
    assert bench.checksum_alu_ops(mode, kernel, streams, rows) == ops
