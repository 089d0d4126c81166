"""Leaf extents with label sizes given as small numpy integers: the product is
taken in Python integers, so that an undersized leaf is still refused (no
GPU: every case ends before a device call)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2002_01935_gb300 import binding  # noqa: E402


@pytest.mark.parametrize("kind", [np.uint8, np.int8, np.int16, np.int32, np.int64])
def test_sizes_of_any_integer_type(kind):
    dims = {l: kind(4) for l in range(8)}  # 4^8 entries a leaf: 0 in 8 bits, and in 16
    labels = [list(range(8)), list(range(8))]
    h = binding.TensorNetwork(labels, dims, [], complex_=False)
    try:
        with pytest.raises(binding.TNError):
            h.set_tensors([torch.zeros(4 ** 8 - 1)] * 2)
        h.set_tensors([torch.zeros(4 ** 8)] * 2)
        assert h._leaf_numel(0) == 4 ** 8
        h._check_strides(1, [0, 0])
        with pytest.raises(binding.TNError):
            h._check_strides(2, [1, 0])
    finally:
        h.close()
