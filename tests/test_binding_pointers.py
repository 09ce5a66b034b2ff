"""The binding's pointer of an argument: what has memory of its own is taken, the rest refused."""
import numpy as np
import pytest

from paper_2607_00579_gb300 import _binding as B


class Interface:
    """An array interface whose data is no address."""
    __array_interface__ = {"version": 3, "shape": (1,), "typestr": "|u1", "data": b"\x07"}


@pytest.mark.parametrize("x", [np.zeros((3, 4)), np.zeros(5, np.float32)[::2], np.zeros(0), np.zeros(2).view(np.recarray)])
def test_arrays(x):
    assert B._ptr(x).value == x.ctypes.data


@pytest.mark.parametrize("x", [np.float64(1.0), np.int64(8), Interface(), 1.5, "x", [1.0]])
def test_others_are_refused(x):
    with pytest.raises(TypeError):
        B._ptr(x)
