"""Host-side ranges of the digit products (no GPU needed): every FP32 sum of a range stays an integer below 2^24.

Digits |d_1| <= 2^7, |d_i| <= 2^6 for i > 1; the pairs (i, j) of one significance i + j, up to i + j = nd + 1, are
summed over a range of K in FP32 and the ranges added in FP64.
"""
import ctypes

import pytest

from paper_2206_07660_gb300 import LIB_PATH


def _pairs_bound(g, nd):
    return sum(2 ** (7 if i == 1 else 6) * 2 ** (7 if g - i == 1 else 6)
               for i in range(1, nd + 1) if 1 <= g - i <= nd)


@pytest.mark.parametrize("nd", [8, 5])
def test_ranges_are_exact_and_complete(nd):
    lib = ctypes.CDLL(LIB_PATH)
    lib.gwdbg_digit_ranges.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    lib.gwdbg_digit_ranges.restype = None
    out = (ctypes.c_int * 4)()
    worst = max(_pairs_bound(g, nd) for g in range(2, nd + 2))
    longest = 0
    for k in list(range(1, 3000)) + [4095, 4096, 4097, 18432, 20000]:
        lib.gwdbg_digit_ranges(k, nd, out)
        block, blocks, per, ranges = out
        assert (blocks - 1) * block < k <= blocks * block
        assert (ranges - 1) * per < blocks <= ranges * per      # none is empty
        terms = min(k, per * block)
        assert terms * worst <= 2 ** 24, k
        longest = max(longest, terms)
    assert longest * worst > 2 ** 23    # and they are not needlessly short
