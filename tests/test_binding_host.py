"""Argument marshalling of the Python binding that needs no GPU: ids."""
import array

import numpy as np
import pytest

ID = bytes(range(100, 116))


@pytest.fixture(scope="module")
def binding():
    from paper_2607_01308_gb300 import _binding
    return _binding


@pytest.mark.parametrize("form", [bytes, bytearray, memoryview, list, tuple,
                                  lambda b: array.array("I", list(b)), lambda b: memoryview(array.array("H", list(b))),
                                  lambda b: np.frombuffer(b, dtype=np.uint8),
                                  lambda b: np.array(list(b), dtype=np.int64),
                                  lambda b: [x - 256 for x in b]])
def test_an_id_is_its_sixteen_entries_whatever_their_type(binding, form):
    arr = binding._id_array([form(ID), ID])
    assert bytes(arr) == ID + ID


@pytest.mark.parametrize("wrong", [ID[:15], ID + b"x", list(ID)[:3], array.array("I", range(4))])
def test_an_id_of_another_length_is_refused(binding, wrong):
    with pytest.raises(ValueError):
        binding._id_array([wrong])


def test_no_ids_still_give_an_array(binding):
    assert len(binding._id_array([])) == 1
