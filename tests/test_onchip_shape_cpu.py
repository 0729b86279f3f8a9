"""Default register bits of the on-chip energy kernel, on CPU: one register bit
only for small complex128 states that leave most SMs without a warp."""
import ctypes

import pytest

sv = pytest.importorskip("paper_2406_03466_gb300")


def reg_bits(n, dtype, slots, kind=0, sms=152):
    r = ctypes.c_int32()
    assert sv.library().sv_debug_onchip_shape(kind, n, dtype, slots, sms, ctypes.byref(r), None) == 0
    return r.value


@pytest.mark.parametrize("n,slots,want", [(2, 1, 1), (4, 33, 1), (4, 1215, 1), (4, 1216, 2), (8, 1, 1), (8, 75, 1),
                                          (8, 76, 2), (9, 1, 2), (9, 33, 2), (10, 2, 2), (11, 1, 2)])
def test_tiny_complex128_batches(n, slots, want):
    assert reg_bits(n, 1, slots) == want


def test_complex64_and_adjoints_keep_theirs():
    for n in (4, 8, 10):
        assert reg_bits(n, 0, 2) == 2
        assert reg_bits(n, 1, 2, kind=3) == 2
