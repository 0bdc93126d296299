"""Shared memory sizes of the elimination launches for tables past 2^31 bytes:
too large to fit, never a small or negative number (no GPU: sizes only)."""
import ctypes

import pytest

from paper_2504_12037_gb300 import tnvan as tv

FIT = 227 * 1024


def _size(name, *args):
    f = getattr(tv.lib(), name)
    f.restype = ctypes.c_int
    return f(*args)


# 4 B x 32 samples x entries: 2^31 at 2^24 entries, a multiple of 2^32 at 2^25
@pytest.mark.parametrize("entries", [1 << 24, (1 << 25) + 16, 50_331_648])
def test_sizes_do_not_wrap(entries):
    b, i = ctypes.c_bool, ctypes.c_int
    assert _size("_ZN5tnvan25general_levels_smem_bytesEiiibi", i(entries), i(0), i(16), b(False), i(1)) > FIT
    assert _size("_ZN5tnvan25general_levels_smem_bytesEiiibi", i(entries // 2), i(0), i(16), b(True), i(3)) > FIT
    assert _size("_ZN5tnvan28general_levels_dJ_smem_bytesEiiiiii", i(entries), i(0), i(0), i(0), i(16), i(7)) > FIT
    # lane groups: rows of 10 floats at 16 lanes a sample
    assert _size("_ZN5tnvan18general_smem_bytesEiiiibb", i(entries * 32 // 10), i(16), i(8), i(16), b(False),
                 b(False)) > FIT
    assert _size("_ZN5tnvan21general_dJ_smem_bytesEiiiiib", i(entries * 32 // 10), i(16), i(100), i(8), i(16),
                 b(False)) > FIT
    assert _size("_ZN5tnvan22general_mom_smem_bytesEiiiib", i(entries), i(16), i(8), i(16), b(False)) > FIT
    # with the tables in global memory nothing but the spins and the cut steps' maxima is left
    assert 0 < _size("_ZN5tnvan28general_levels_dJ_smem_bytesEiiiiii", i(entries), i(entries), i(entries), i(64), i(16),
                     i(0)) <= FIT


def test_sizes_of_small_tables():
    b, i = ctypes.c_bool, ctypes.c_int
    assert _size("_ZN5tnvan25general_levels_smem_bytesEiiibi", i(100), i(3), i(16), b(True), i(3)) == 128 * 203 + 640
    assert _size("_ZN5tnvan28general_levels_dJ_smem_bytesEiiiiii", i(70), i(30), i(20), i(5), i(16), i(7)) == \
        128 * 125 + 640
