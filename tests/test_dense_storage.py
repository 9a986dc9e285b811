"""Shared memory of a cell: what it may cost in cells an SM holds."""
import json

import pytest

from paper_2111_07436_gb300 import camp, workloads as w

BLOCK = 227 * 1024 - 256  # dynamic shared memory of one block


def gas(n, processes=1.0):
    part = [max(1, round(k * n * processes / 72)) for k in (112, 28, 28, 9, 9)]
    return w.gas_mechanism(f"gas-{n}", n, *part, seed=1000 + n)


def resident(nbytes, warps):
    """Cells of one warp each that an SM's 228 KB hold, up to `warps`."""
    return max((c * min(warps // c, 228 * 1024 // (c * nbytes + 1024)) for c in (1, 2, 3, 4) if c * nbytes <= BLOCK),
               default=0)


@pytest.mark.parametrize("n,form,cells", [(117, "fp64", 3), (73, "mixed", 12), (91, "mixed", 8)])
def test_halves_cost_no_resident_cells(n, form, cells):
    """The odd halves of the forcing sums are left out where an SM holds more
    cells without them."""
    inf = camp.Mechanism(json.dumps(gas(n)), device=False).info
    assert resident(getattr(inf, "smem_per_cell_" + form), 8 if form == "fp64" or n > 128 else 12) == cells
