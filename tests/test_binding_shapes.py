"""Array arguments of the binding: any object with a data pointer, whatever sequence its shape is."""
import numpy as np
import pytest
import torch

from paper_1405_2728_gb300 import mm


class Array:
    """What another library's tensor looks like: a pointer, a dtype, and a shape that is a list."""

    def __init__(self, a):
        self.a, self.shape, self.dtype = a, list(a.shape), a.dtype

    def data_ptr(self):
        return self.a.ctypes.data

    def is_contiguous(self):
        return self.a.flags.c_contiguous


def test_shapes_are_compared_as_sequences():
    a = np.zeros((3, 2, 4, 5))
    for x in (Array(a), torch.from_numpy(a)):
        for shape in ((3, 2, 4, 5), [3, 2, 4, 5]):
            assert mm._ptr(x, np.float64, shape).value == a.ctypes.data
        for shape in ((3, 2, 5, 4), (3, 2, 4), ()):
            with pytest.raises(ValueError):
                mm._ptr(x, np.float64, shape)
        with pytest.raises(TypeError):
            mm._ptr(x, np.float32, (3, 2, 4, 5))
