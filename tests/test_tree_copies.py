"""Copies of a draft tree that has been handed to the library (no GPU needed: only addresses are taken)."""
import copy
import ctypes
import dataclasses
import pickle

import pytest
import torch


def _tree():
    from paper_2601_07353_b200.talon import Tree
    t = Tree(*(torch.zeros(2, dtype=torch.int32) for _ in range(8)))
    t.address()                                          # as every call of the library does
    return t


def _arrays(tree):
    from paper_2601_07353_b200.talon import TalonTreeStruct
    s = TalonTreeStruct.from_address(tree.address())
    return [ctypes.cast(getattr(s, n), ctypes.c_void_p).value for n, _ in TalonTreeStruct._fields_]


@pytest.mark.parametrize("how", [copy.deepcopy, copy.copy, dataclasses.replace, lambda t: pickle.loads(pickle.dumps(t))],
                         ids=["deepcopy", "copy", "replace", "pickle"])
def test_a_copy_points_at_its_own_arrays(how):
    tree = _tree()
    other = how(tree)
    for t in (other, tree):
        assert _arrays(t) == [getattr(t, f.name).data_ptr() for f in dataclasses.fields(t)]
    other.token = torch.ones(2, dtype=torch.int32)
    assert _arrays(other)[1] == other.token.data_ptr() and _arrays(tree)[1] == tree.token.data_ptr()
