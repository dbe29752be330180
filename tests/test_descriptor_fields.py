"""The batched calls' descriptors as the wrappers pack them: the bytes of the ctypes structures
that mirror the C ones, field by field, and of the sizes the wrappers' values have."""

import ctypes
import random

import pytest

from paper_2609_11687_gb300 import kashin as kd

STRUCTS = [kd.KdMatrix, kd.KdFoldMat, kd.KdFoldMatF16, kd.KdPMat, kd.KdPlane, kd.KdRecMat]


@pytest.mark.parametrize("cls", STRUCTS)
@pytest.mark.parametrize("count", [1, 3, 32])
def test_packed_bytes(cls, count):
    rng = random.Random(count)
    arr = (cls * count)()
    vals = []
    for d in arr:
        for name, t in cls._fields_:
            v = rng.choice((0, 1, rng.getrandbits(47), 2 ** 63 - 1)) if t is not ctypes.c_uint64 else rng.getrandbits(64)
            setattr(d, name, v)
            vals.append(v)
    assert kd._pack(cls, count, vals) == bytes(arr)


def test_a_missing_value_is_refused():
    with pytest.raises(Exception):
        kd._pack(kd.KdPMat, 2, [0] * 7)
