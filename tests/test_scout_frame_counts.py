"""The scout binding's frame counts: any sequence of integers, as ctypes takes it.

Byte strings are sequences of small integers, and counts beyond 32 bits are
refused with VisCacheError like every other size the library does not take."""
import array
import ctypes
import types

import numpy as np
import pytest
import torch

from paper_2608_24063_gb300 import viscache as vc


@pytest.mark.parametrize("counts", [[64, 3], (64, 3), range(1, 4), np.array([64, 3]), np.array([64, 3], dtype=np.uint8),
                                    torch.tensor([64, 3]), b"\x40\x03", b"\x40\x03\x01\x01", bytearray(b"\x40\x03"),
                                    array.array("q", [64, 3]), [], [-1], [True, 2], [np.int64(3)], [2 ** 31],
                                    [2 ** 32 + 64]], ids=str)
def test_counts_are_what_ctypes_makes_of_them(counts):
    want = (ctypes.c_int32 * len(counts))(*counts)
    got = vc._frame_counts(counts)
    assert isinstance(got, ctypes.c_int32 * len(counts)) and got[:] == want[:]


@pytest.mark.parametrize("counts", [[64.0], "ab", np.array([64.0]), [None]], ids=str)
def test_what_is_no_integer_is_a_type_error(counts):
    with pytest.raises(TypeError):
        vc._frame_counts(counts)


@pytest.mark.parametrize("counts", [[2 ** 31], [0], [-5], [3, 2 ** 31 + 7]], ids=str)
def test_sizes_the_library_does_not_take_are_its_error(counts):
    H = types.SimpleNamespace(shape=(64, 512))
    with pytest.raises(vc.VisCacheError):
        vc.viscache_scout_mmr(H, None, counts)
