"""How the binding hands host lengths and spans to the library: the short way for lists of
integers takes what numpy's conversion takes, gives the same array and refuses the same."""
import ctypes

import numpy as np
import pytest

from paper_2604_05650_b200 import binding


def _read(addr, n):
    return list((ctypes.c_int32 * n).from_address(addr)) if n else []


@pytest.mark.parametrize("value,nested", [
    ([5, 7], False), ([True, 2], False), ([np.int32(3), np.int64(4)], False), ([1.0, 2.9], False), ((8, 9), False),
    (np.asarray([1, 2, 3], np.int64), False), (np.arange(8, dtype=np.int32)[::2], False), ([-1, 2**31 - 1], False),
    ([[0, 3], [4, 9]], True), ([(0, 3), (4, 9)], True), ([0, 3, 4, 9], True), ([[0.0, 3.5]], True),
    (np.asarray([[0, 3], [4, 9]], np.int32), True), (np.asarray([[0, 3], [4, 9]], np.int32).T, True), ([[[0, 3]]], True),
    ([np.asarray([0, 3]), np.asarray([4, 9])], True), ([], False),
])
def test_same_as_numpy(value, nested):
    want = np.ascontiguousarray(np.asarray(value, dtype=np.int32)).ravel()
    addr, n, _keep = binding._host_i32(value, nested)
    assert n == want.size and _read(addr, n) == want.tolist()


class _Index:
    """An integer to array.array, nothing to numpy."""
    def __index__(self):
        return 3

    def __int__(self):
        raise TypeError("no")


@pytest.mark.parametrize("value,nested", [
    ([{0, 3}], True), ([{0: 1, 3: 2}], True), ([b"ab"], True), ([frozenset([4, 9]), [0, 3]], True),
    ([_Index(), 2], False), ([[_Index(), 2]], True), ([iter([0, 3])], True),
])
def test_what_numpy_refuses_stays_refused(value, nested):
    """Rows that are not sequences, and elements that only look like integers, do not slip
    through the short way (a set's order is not the caller's)."""
    with pytest.raises((OverflowError, ValueError, TypeError)) as want:
        np.asarray(value, dtype=np.int32)
    with pytest.raises(want.type):
        binding._host_i32(value, nested)


@pytest.mark.parametrize("value,nested", [([2**31], False), ([[0, 2**40]], True), (["x"], False), ([[0, 1], [2]], True),
                                          ([None], False)])
def test_refused_as_before(value, nested):
    with pytest.raises((OverflowError, ValueError, TypeError)) as want:
        np.asarray(value, dtype=np.int32)
    with pytest.raises(want.type):
        binding._host_i32(value, nested)
