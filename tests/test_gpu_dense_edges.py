"""The dense block's factorisation and triangular solves at the edges of
their tiles (32-row slots, 8-column panels, 4-pivot rounds) on one warp and on
64 threads a cell, and the block-arrow form at the edges of its unrolled
particle solves (8 and 16 species a particle), against the oracle."""
import json

import numpy as np
import pytest

import oracle
from paper_2111_07436_gb300 import camp, workloads as w
from tests import mechs, parity

pytestmark = pytest.mark.gpu


def _gas(n):
    part = [max(1, round(k * n / 72)) for k in (112, 28, 28, 9, 9)]
    return w.gas_mechanism(f"gas-{n}", n, *part, seed=1000 + n)


# species of the mechanism: dense blocks of 8..109 rows (the block's size is
# the mechanism's; the sizes here leave remainders of 0..7 rows in a panel and
# blocks of one to four slots)
@pytest.mark.parametrize("variant,tol", [(camp.VARIANT_FP64, 1e-10), (camp.VARIANT_MIXED, 1e-4)])
@pytest.mark.parametrize("lanes", [32, 64])
@pytest.mark.parametrize("n", [10, 12, 24, 38, 40, 42, 44, 60, 76, 80, 82, 84, 86, 100, 116, 126])
def test_lu_solve_at_tile_edges(cuda, n, lanes, variant, tol):
    import torch
    mj = _gas(n)
    gm, om = camp.Mechanism(json.dumps(mj)), oracle.Mechanism(json.dumps(mj))
    gm.set_lanes(lanes)
    y, env = w.cells(mj, 5, seed=n)
    b = np.random.default_rng(n).normal(size=y.shape)
    gamma = 0.1
    x, st = gm.lu_solve(torch.tensor(y, device=cuda), torch.tensor(env, device=cuda), gamma,
                        torch.tensor(b, device=cuda), variant=variant)
    x, st = x.cpu().numpy(), st.cpu().numpy()
    assert (st == 0).all()
    u = 2.0 ** -53 if variant == camp.VARIANT_FP64 else 2.0 ** -24
    for c in range(len(y)):
        kf, kr = om.rate_constants(env[c])
        M = np.eye(gm.n) - gamma * om.jacobian(kf, kr, y[c], env[c])
        xo = oracle.dense_lu_solve(M, b[c])
        r = np.linalg.norm(M @ x[c] - b[c]) / (np.linalg.norm(M, np.inf) * np.linalg.norm(x[c], np.inf))
        assert r <= tol
        assert np.linalg.norm(x[c] - xo) / np.linalg.norm(xo) <= max(tol * 1e3, 10 * np.linalg.cond(M) * u)


def _particles(n_phase, n_particles):
    """n_phase species a particle: a transferred species and a chain behind it."""
    names = [f"A{i}" for i in range(n_phase)]
    rx = [mechs.photolysis("G1", {"G2": 1.0}, value=1e-3), mechs.henry("G1", "A0", H298=2e3 / 101325.0, alpha=0.2),
          mechs.henry("G2", "A1", H298=1e2 / 101325.0, alpha=0.1)]
    rx += [mechs.condensed_arrhenius({names[i]: 1}, {names[i + 1]: 1.0}, A=10.0 ** -(1 + i % 3))
           for i in range(n_phase - 1)]
    mj = json.loads(mechs.mech(["G1", "G2"], rx, phase=names, sections=n_particles))
    mj["aerosol"].update(representation="particles", solver="block_arrow")
    return mj


@pytest.mark.parametrize("variant", [camp.VARIANT_FP64, camp.VARIANT_MIXED])
@pytest.mark.parametrize("n_phase", [2, 7, 8, 9, 15, 16])
def test_block_arrow_species_per_particle(cuda, n_phase, variant):
    import torch
    mj = _particles(n_phase, 37)
    gm, om = camp.Mechanism(json.dumps(mj)), oracle.Mechanism(json.dumps(mj))
    assert gm.info.block_arrow == 1
    y0, env = w.cells(mj, 6, seed=n_phase)
    yo, so, _ = om.solve(y0, env, 60.0, 1e-4, 1e-5)
    assert (so == 0).all()
    ty = torch.tensor(y0, device=cuda)
    st = gm.solve(ty, torch.tensor(env, device=cuda), 60.0, 1e-4, 1e-5, variant=variant)
    assert (st.cpu().numpy() == 0).all()
    parity.check(om, y0, env, 60.0, 1e-4, 1e-5, ty.cpu().numpy(), yo)
