"""f(y) by a lane a cell or by a warp a cell: the rule against the measured
times of both on 152 SMs, and the same values on both sides of its lines."""
import ctypes
import json

import numpy as np
import pytest

from paper_2111_07436_gb300 import build, camp, workloads as w

# processes, cells, microseconds of a warp a cell, of a lane a cell
MEASURED = [(12, 1024, 33.5, 45.7), (12, 3072, 90.8, 45.7), (12, 4864, 139.9, 45.7), (12, 65536, 1595, 105),
            (61, 4864, 156, 253), (61, 8192, 238, 267), (61, 9728, 273, 267), (61, 12288, 355, 289),
            (186, 12288, 756, 822), (186, 13500, 840, 824), (186, 19456, 1187, 903), (186, 19488, 1191, 1613),
            (186, 26624, 1604, 1756), (186, 32768, 1967, 1758), (186, 38912, 2334, 1774), (186, 40000, 2396, 2584),
            (186, 65536, 3909, 3475), (222, 12288, 1008, 1057), (222, 13500, 1103, 1065), (222, 19488, 1569, 2053),
            (222, 65536, 5176, 4444)]


@pytest.mark.parametrize("processes,cells,warp,lane", MEASURED)
def test_rule_takes_the_faster_kernel(processes, cells, warp, lane):
    build.build()
    rule = ctypes.CDLL(build.LIB).camp_forcing_by_lanes
    rule.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    assert rule(processes, cells, 152) == (lane < warp)


def test_four_warps_of_rates_fit_an_sm():
    build.build()
    rule = ctypes.CDLL(build.LIB).camp_forcing_by_lanes
    rule.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_int]
    assert rule(224, 65536, 152) and not rule(225, 65536, 152)


@pytest.mark.gpu
@pytest.mark.parametrize("mech,cells", [("small", 2113), ("small", 2305), ("gas", 13537), ("gas", 19489),
                                        ("gas", 38881), ("gas", 40001)])
def test_values_on_both_sides(cuda, mech, cells):
    import torch
    mj = {"small": w.small_gas_mechanism, "gas": w.large_gas_mechanism}[mech]()
    m = camp.Mechanism(json.dumps(mj))
    y, env = w.cells(mj, cells, seed=12)
    ty, te = torch.tensor(y, device="cuda"), torch.tensor(env, device="cuda")
    big = m.forcing(ty, te).cpu().numpy()
    part = 500  # far below the line: a warp a cell
    for lo in (0, cells // 2, cells - part):
        few = m.forcing(ty[lo:lo + part].contiguous(), te[lo:lo + part].contiguous()).cpu().numpy()
        assert np.array_equal(big[lo:lo + part], few)
