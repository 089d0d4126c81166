"""Tree lists of any rows: tuples, lists and numpy rows, changed in place or
in a new list that happens to have the address of a freed one (no GPU)."""
import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2002_01935_gb300 import binding  # noqa: E402

ROWS = np.array([[0, 1], [2, 3]])


def test_row_in_place_of_a_tuple():
    pairs = [(0, 1), (2, 3)]
    assert binding._tree(pairs).tolist() == [0, 1, 2, 3]
    pairs[0] = np.array([1, 0])
    assert binding._tree(pairs).tolist() == [1, 0, 2, 3]
    assert binding._tree(pairs).tolist() == [1, 0, 2, 3]


def test_new_list_of_rows_after_a_list_of_tuples():
    first, second = ROWS
    reused = 0
    for _ in range(50):
        pairs = [(0, 1), (2, 3)]
        binding._tree(pairs)
        address = id(pairs)
        del pairs
        rows = [second, first]
        reused += id(rows) == address
        assert binding._tree(rows).tolist() == [2, 3, 0, 1]
        del rows
        binding._tree_cache.clear()
    assert reused


def test_rows_of_torch_tensors():
    import torch
    pairs = [(0, 1), (2, 3)]
    binding._tree(pairs)
    pairs[1] = torch.tensor([3, 2])
    assert binding._tree(pairs).tolist() == [0, 1, 3, 2]


def test_lists_and_tuples_with_other_values():
    pairs = [(0, 1), (2, 3)]
    binding._tree(pairs)
    pairs[1] = [3, 2]
    assert binding._tree(pairs).tolist() == [0, 1, 3, 2]
    pairs[1] = (2, 3)
    assert binding._tree(pairs).tolist() == [0, 1, 2, 3]
