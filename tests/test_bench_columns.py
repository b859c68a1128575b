"""bench.py's column-storage model (no GPU): which storage each product's bytes are counted
on, by value type, row shape, entries and row length, and the bytes of block offsets."""
import os
import sys
import types

import numpy as np
import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("shape,value_type,rows,length,expect", [
    ("16x2", "f32", 10000, 200, "block"), ("16x2", "bf16", 10000, 200, "block"),
    ("16x1", "f64", 10000, 200, False), ("16x2", "f64", 10000, 200, False),
    ("32x1", "f32", 10000, 200, False), ("16x2/16-bit", "f32", 10000, 200, True),
    ("16x1/16-bit", "f64", 10, 3, True),
    # below 2^20 stored entries: 4681 rows of 217 entries, stored as 224, are above
    ("16x2", "f32", 4681, 224, False), ("16x2", "f32", 4682, 217, "block"),
    # fewer than 64 stored entries per row, and more than 43776 rows
    ("16x2", "f32", 43777, 56, False), ("16x2", "f32", 43777, 57, "block"),
    ("16x2", "f32", 43776, 56, "block"), ("16x2", "f32", 30000, 40, "block")])
def test_stored_columns(shape, value_type, rows, length, expect):
    assert bench.stored_columns(shape, value_type, np.full(rows, length)) == expect


def test_block_bytes_by_hand():
    P = types.SimpleNamespace(m=3, n=5, nnz=64)
    # FP32 values, 2-byte offsets, one 4-byte base per 64 entries, a 4-byte index per row;
    # row pointers, output and input vector
    a = 64 * (4 + 2) + 4 + 3 * 4 + 4 * 4 + 3 * 4 + 5 * 4
    at = 64 * (4 + 2) + 4 + 5 * 4 + 6 * 4 + 5 * 4 + 3 * 4
    assert bench.spmv_bytes(P, "f32", "block", "block") == pytest.approx(0.5 * (a + at))


def test_both_directions_of_a_batch():
    rng = np.random.default_rng(0)
    Ps = []
    for m, n, L in ((6000, 22000, 100), (7000, 22000, 100)):
        Ps.append(types.SimpleNamespace(m=m, n=n, row_ptr=np.arange(m + 1) * L,
                                        col_idx=rng.integers(0, n, m * L)))
    # rows of 104 stored entries; 44000 columns of about 30
    assert bench.matrix_columns(Ps, "f32", "16x2", "16x2") == ("block", False)
    assert bench.matrix_columns(Ps[:1], "f32", "16x2", "16x2") == (False, False)
