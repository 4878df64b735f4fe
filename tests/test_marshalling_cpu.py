"""Host index arrays of the binding: every form a caller may pass reaches the library as the same values."""
import ctypes

import numpy as np
import pytest

from paper_2608_27206_gb300 import pace as P


@pytest.mark.parametrize("conv,width", [(P._i32, ctypes.c_int32), (P._i64, ctypes.c_int64)])
@pytest.mark.parametrize("form", [list, tuple, lambda a: np.asarray(a, np.int32), lambda a: np.asarray(a, np.int64),
                                  lambda a: np.repeat(np.asarray(a, np.int32), 2)[::2], lambda a: [np.int32(x) for x in a],
                                  lambda a: [float(x) for x in a], lambda a: np.asarray(a, np.float64)])
def test_index_arrays(conv, width, form):
    want = [0, 7, 2156, 1 << 20]
    owner, address, n = conv(form(want))
    assert n == 4 and list((width * n).from_address(address)) == want
    assert [int(x) for x in owner] == want


def test_index_arrays_out_of_range_and_empty():
    with pytest.raises(OverflowError):
        P._i32([1 << 31])
    assert P._i32([])[2] == 0


def test_patch_counts():
    for h, w in ([[28], [42]], [[28, 2156, 14], [42, 3836, 27]]):
        owners = P._i32(h)[0], P._i32(np.asarray(w, np.int32))[0]
        assert P._n_patches(*owners) == sum(a // 14 * (b // 14) for a, b in zip(h, w))
    with pytest.raises(ValueError):
        P._n_patches(P._i32([28, 28])[0], P._i32([28])[0])
