"""Which form the FP32 flux pass takes (CPU; a rule on sizes): two ranges of columns
in turn only where neighbouring ranges share the 32-byte sectors of the flux sums
(velocity rows that are no multiple of four), one CTA walks a tile's rows and the
array exceeds the L2.  Elsewhere that form is the slower one, by up to a tenth."""
import ctypes
import os

import pytest

from paper_2604_09984_gb300 import ugks as U


@pytest.fixture(scope="module")
def rule():
    if not os.path.exists(U.LIB_PATH):
        import __graft_entry__
        __graft_entry__.build()
    f = U.load()["_ZN4ugks10flux_pairsEmii"]        # ugks::flux_pairs(unsigned long, int, int)
    f.restype, f.argtypes = ctypes.c_bool, (ctypes.c_size_t, ctypes.c_int, ctypes.c_int)
    return f


@pytest.mark.parametrize("nvx", [21, 22, 24, 25, 28, 31, 33, 36, 40, 48])
@pytest.mark.parametrize("nsplit", [1, 2, 7])
@pytest.mark.parametrize("items,large", [(9216 * 1104, False), (15_000_000, False), (15_000_016, True), (52200 * 1104, True)])
def test_pairs_where_ranges_share_sectors(rule, items, large, nsplit, nvx):
    assert rule(items, nvx, nsplit) == (large and nsplit == 1 and nvx % 4 != 0)
