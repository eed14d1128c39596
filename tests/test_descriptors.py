"""The descriptor arrays take what a ctypes structure's fields take: Python and
NumPy integers of every width, wrapped to the field; nothing that is not an
integer, and no row of another length."""
import ctypes

import numpy as np
import pytest

from paper_1509_02308_gb300 import capi as C
from paper_1509_02308_gb300.workloads import Geom

INTS = [0, 1, True, 7, -1, 2**31, 2**32, 2**33 + 5, 2**64, 2**70, np.int8(-1), np.int32(3), np.uint32(3),
        np.int64(3), np.uint64(2**63), np.array(3)]
OTHERS = [1.0, 1.5, "1", None, [1], np.float32(2), np.bool_(True)]


@pytest.mark.parametrize("v", INTS, ids=repr)
def test_integers_wrap_as_ctypes_fields_do(v):
    def same(got, want):
        assert bytes(got) == bytes(want)

    same(C.pair_array([(v, 1), (2, v)]), (C.Pair * 2)(C.Pair(v, 1), C.Pair(2, v)))
    same(C.trace_array([(None, v, v, v, v)]), (C.Trace * 1)(C.Trace(None, v, v, v, v)))
    same(C.geom_array([Geom(v, v, v, v, v, 9)]), (C.Geom * 1)(C.Geom(v, v, v, v, v, 0, 9)))


@pytest.mark.parametrize("v", OTHERS, ids=repr)
def test_anything_else_is_refused(v):
    for pairs in ([(v, 0)], [(1, 2), (0, v)]):
        with pytest.raises(TypeError):
            C.pair_array(pairs)
    for at in range(1, 5):
        row = [None, 1, 1, 1, 1]
        row[at] = v
        with pytest.raises(TypeError):
            C.trace_array([tuple(row)])
    for at in range(5):
        row = [4096, 32, 4, 32, 0]
        row[at] = v
        with pytest.raises(TypeError):
            C.geom_array([Geom(*row, 1)])


def test_rows_of_another_length_are_refused():
    for pairs in ([(1, 2, 3)], [(1, 2, 3), (1, 2, 3)], [(1,)], [(1, 2, 3, 4)]):
        with pytest.raises(ValueError):
            C.pair_array(pairs)
    with pytest.raises(TypeError):
        C.pair_array([1, 2])
    assert ctypes.sizeof(C.pair_array([])) == ctypes.sizeof(C.Pair)
