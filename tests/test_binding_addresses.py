"""The pointers that a call takes from its buffers, without a GPU."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1710_08576_gb300 import _binding


def _read(seq):
    at, keep = _binding._addresses(seq)
    return list((ctypes.c_uint64 * len(seq)).from_address(at))


def test_tensors_arrays_integers_and_missing_buffers():
    a, b = torch.zeros(8, dtype=torch.int8), torch.zeros(9, dtype=torch.int16)
    n = np.zeros(4, np.int8)
    assert _read([a, b[1:]]) == [a.data_ptr(), b.data_ptr() + 2]
    assert _read((a, None, 4096, n)) == [a.data_ptr(), 0, 4096, n.ctypes.data]
    assert _binding._addresses(None) == (None, None)


@pytest.mark.parametrize("lazy", [iter, lambda s: (t for t in s), lambda s: map(lambda t: t, s)])
def test_iterators_are_refused(lazy):
    """A buffer that only the iterator holds is freed, and may be given to another tensor, before the
    kernel that was given its address has run."""
    with pytest.raises(TypeError):
        _binding._addresses(lazy([torch.zeros(8, dtype=torch.int8)]))
