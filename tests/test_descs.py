"""make_descs packs entries of plain numbers in one call; every other entry, and
every number out of its field's range, takes the general path.  Both give the
descriptors that field-by-field construction gives."""
import ctypes

import numpy as np
import pytest

from paper_2007_10752_gb300 import tdes


def _by_field(entries):
    arr = (tdes.Desc * max(1, len(entries)))()
    for i, (mode, key, iv, ip, op, n) in enumerate(entries):
        arr[i] = tdes.Desc(mode, key, iv & (2**64 - 1), tdes._ptr(ip), tdes._ptr(op), n)
    return bytes(arr)


PLAIN = [(4, 7, 2**64 - 1, 2**63 + 16, 8, 4096), [0, 2**32 - 1, 0, 0, 0, 0]]


@pytest.mark.parametrize("entries", [
    [], PLAIN, PLAIN * 700,
    [(1, 2, -1, 8, 16, 8)], [(1, 2, 2**65 + 3, 8, 16, 8)], [(-1, 2**32 + 5, 0, 8, 16, 2**64 + 8)],
    [(0, 1, 2, np.zeros(8, np.uint8), None, 8)], [(True, 1, 2, 8, 8, 8)],
], ids=["empty", "plain", "many", "negative_iv", "wide_iv", "wide_fields", "array", "other_ints"])
def test_packed_equals_by_field(entries):
    arr, n = tdes.make_descs(iter(entries))
    assert n == len(entries) and bytes(arr) == _by_field(entries)
    assert ctypes.sizeof(arr) == ctypes.sizeof(tdes.Desc) * max(1, n)


@pytest.mark.parametrize("entries", [[(0, 1, 2, 8, 16)], [(0, 1, 2, 8, 16), (0, 1, 2, 8, 16, 8, 9)]])
def test_wrong_length_refused(entries):
    with pytest.raises(ValueError):
        tdes.make_descs(entries)
