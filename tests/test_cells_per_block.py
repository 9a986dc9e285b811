"""Cells a block of the solve takes by default, from the blocks an SM holds at
each count: one when the device is free for them at that, else the count with
the most resident cells."""
import ctypes

import pytest

from paper_2111_07436_gb300 import build

GAS72 = (11, 5, 4, 3)  # blocks of 1..4 cells on an SM: 11, 10, 12, 12 cells


@pytest.mark.parametrize("blocks,cells,beside,expected", [
    (GAS72, 1, 0.0, 1), (GAS72, 256, 0.0, 1), (GAS72, 1672, 0.0, 1), (GAS72, 1673, 0.0, 3),
    (GAS72, 256, 0.8, 1), (GAS72, 256, 0.9, 3), (GAS72, 256, 31 * 256 / 1672, 3), (GAS72, 1, 1.0, 3),
    ((6,), 100000, 5.0, 1), ((4, 4, 2, 2), 100000, 0.0, 2), ((8, 4, 2, 2), 10 ** 9, 0.0, 1)])
def test_default_count(blocks, cells, beside, expected):
    build.build()
    rule = ctypes.CDLL(build.LIB).camp_default_cells_per_block
    rule.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_longlong, ctypes.c_int, ctypes.c_double]
    per_sm = (ctypes.c_int * 5)(0, *blocks)
    assert rule(per_sm, len(blocks), cells, 152, beside) == expected
