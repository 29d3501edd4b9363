"""Label arrays as the binding hands them to the C ABI: one C int per label, for
every kind of sequence."""
import array

import numpy as np
import pytest

from paper_2104_10523_gb300 import tnq


@pytest.mark.parametrize("labels", [
    [3, 0, 2, 1], (3, 0, 2, 1), np.array([3, 0, 2, 1]), np.array([3, 0, 2, 1], np.int8), np.array([3.0, 0.0, 2.0, 1.0]),
    array.array("q", [3, 0, 2, 1]), bytes([3, 0, 2, 1]), bytearray([3, 0, 2, 1]), memoryview(bytes([3, 0, 2, 1])),
    "3021"], ids=lambda v: type(v).__name__)
def test_one_int_per_label(labels):
    assert tnq._labels(labels) == np.array([3, 0, 2, 1], np.int32).tobytes()


def test_empty_and_wide():
    assert tnq._labels([]) == b"" and tnq._labels(b"") == b""
    assert tnq._labels([2 ** 32 + 5, -1]) == np.array([5, -1], np.int32).tobytes()  # as a C int array takes them
