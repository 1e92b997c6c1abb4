"""The index of the tube pass's DFT tables: r kh mod nh from an FP32 reciprocal, corrected by one
step either way, is exact for every length the tile form takes (nh < 256)."""
import numpy as np


def test_table_index_is_exact():
    for nh in range(1, 256):
        rnh = np.float32(1) / np.float32(nh)
        x = np.arange(nh)[:, None] * np.arange(nh // 2 + 1)[None, :]
        m = x - (x.astype(np.float32) * rnh).astype(np.int32) * nh
        m = np.where(m < 0, m + nh, m)
        m = np.where(m >= nh, m - nh, m)
        assert np.array_equal(m, x % nh), nh
