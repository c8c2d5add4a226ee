"""The binding's check of buffer types: a tensor dtype only, by its full name."""
import numpy as np
import pytest
import torch

from paper_2608_22646_gb300 import _buf


class _Foreign:
    """An array of another library: a numpy dtype on an object with PyTorch's
    method names."""

    def __init__(self, dtype):
        self.dtype = np.dtype(dtype)

    def is_contiguous(self):
        return True

    def data_ptr(self):
        return 4096


@pytest.mark.parametrize("dtype", ["float32", "int32"])
def test_foreign_dtypes_are_refused(dtype):
    for _ in range(2):  # the second look finds the dtype's name remembered
        with pytest.raises(ValueError):
            _buf(_Foreign(dtype), "x", dtype)
    t = torch.zeros(4, dtype=getattr(torch, dtype))
    assert _buf(t, "x", dtype) == t.data_ptr()
