"""f(y) by a warp a cell and by a lane a cell (large batches): the same values
bit for bit, on both sides of the rule's line and on ragged last warps."""
import json

import numpy as np
import pytest

from paper_2111_07436_gb300 import camp, workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mech,cells", [("small", 4873), ("small", 4877), ("gas", 12591), ("gas", 12607),
                                        ("variety", 9999), ("variety", 13033), ("sections", 13100)])
def test_forcing_of_large_batches(cuda, mech, cells):
    import torch
    mj = {"small": w.small_gas_mechanism, "gas": w.large_gas_mechanism, "variety": w.process_variety_mechanism,
          "sections": lambda: dict(w.multiphase_mechanism(), aerosol={"phase": "aqueous", "sections": 2})}[mech]()
    m = camp.Mechanism(json.dumps(mj))
    assert m.info.lanes_per_cell == 32
    y, env = w.cells(mj, cells, seed=11)
    y[:, -1] = 0.0
    ty, te = torch.tensor(y, device="cuda"), torch.tensor(env, device="cuda")
    big = m.forcing(ty, te).cpu().numpy()
    part = 1000  # far below the line: a warp a cell
    for lo in (0, cells // 2, cells - part):
        few = m.forcing(ty[lo:lo + part].contiguous(), te[lo:lo + part].contiguous()).cpu().numpy()
        assert np.array_equal(big[lo:lo + part], few)
