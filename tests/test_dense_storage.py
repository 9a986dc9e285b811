"""Shared memory of a cell: what the dense block's row padding and the odd
halves of the forcing sums may cost in cells an SM holds, where the block
starts, and the factorisation on each of the strides that follow."""
import json

import numpy as np
import pytest

import oracle
from paper_2111_07436_gb300 import camp, workloads as w

BLOCK = 227 * 1024 - 256  # dynamic shared memory of one block


def gas(n, processes=1.0):
    part = [max(1, round(k * n * processes / 72)) for k in (112, 28, 28, 9, 9)]
    return w.gas_mechanism(f"gas-{n}", n, *part, seed=1000 + n)


def cut():
    """A 117-species mechanism of so many processes that an FP64 cell fits a
    block of threads with 91 values a row of its 91-row block, not with 92."""
    mj = gas(117)
    room = BLOCK - camp.Mechanism(json.dumps(mj), device=False).info.smem_per_cell_fp64
    extra = dict(next(r for r in mj["reactions"] if r["type"] == "ARRHENIUS"))
    extra["A"] *= 1e-12
    mj["reactions"] += [extra] * (room // 16 + 20)  # a rate constant and a rate term each
    return mj


def resident(nbytes, warps):
    """Cells of one warp each that an SM's 228 KB hold, up to `warps`."""
    return max((c * min(warps // c, 228 * 1024 // (c * nbytes + 1024)) for c in (1, 2, 3, 4) if c * nbytes <= BLOCK),
               default=0)


def compact(m, elem):
    """Bytes of a one-warp gas cell whose block has odd rows of no more than
    one value's padding, and no halves."""
    s, inf = m.structure(), m.info
    D, n = inf.dense_block, inf.n_species
    d = n - D
    sparse = sum((i < d) or (int(j) < d) for i in range(n)
                 for j in s["lu_colidx"][s["lu_rowptr"][i]:s["lu_rowptr"][i + 1]])
    al = lambda b: (b + 15) & ~15
    assert 8 * inf.n_rxn >= elem * n
    return al(8 * n) + 2 * al(8 * inf.n_rxn) + al(elem * (((sparse + 3) & ~3) + D * (D | 1)))


@pytest.mark.parametrize("n,form,cells", [(117, "fp64", 3), (73, "mixed", 12), (91, "mixed", 8)])
def test_halves_cost_no_resident_cells(n, form, cells):
    """The odd halves of the forcing sums are left out where an SM holds more
    cells without them."""
    inf = camp.Mechanism(json.dumps(gas(n)), device=False).info
    assert resident(getattr(inf, "smem_per_cell_" + form), 8 if form == "fp64" or n > 128 else 12) == cells


def test_gas_mechanisms_keep_their_resident_cells():
    """FP64 cells: at least three quarters of those without padding and halves
    (a count that halves costs 1.2 times the time, one that loses a cell of
    four or more none); FP32 cells, less sensitive: two thirds."""
    for n in range(24, 193):
        m = camp.Mechanism(json.dumps(gas(n)), device=False)
        inf = m.info
        assert inf.lanes_per_cell == 32
        assert 4 * resident(inf.smem_per_cell_fp64, 8) >= 3 * resident(compact(m, 8), 8), n
        warps = 12 if n <= 128 else 8
        assert 3 * resident(inf.smem_per_cell_mixed, warps) >= 2 * resident(compact(m, 4), warps), n


@pytest.mark.parametrize("n,processes", [(220, 1.1), (220, 1.2), (234, 1.0), (242, 0.9), (250, 1.1), (254, 1.0)])
def test_block_is_not_cut_where_it_fits(n, processes):
    """The block is the smallest tail with a fill of three quarters, at most
    128 rows, also near the limits of a block's shared memory (with the partial
    sums there are) and of the packed offsets."""
    m = camp.Mechanism(json.dumps(gas(n, processes)), device=False)
    s = m.structure()
    for d in range(n - 7):
        fill = sum(int((s["lu_colidx"][s["lu_rowptr"][i]:s["lu_rowptr"][i + 1]] >= d).sum()) for i in range(d, n))
        if fill >= 0.75 * (n - d) ** 2:
            break
    assert m.info.dense_block == min(n - d, 128)


def test_block_is_cut_where_only_compact_rows_fit():
    inf = camp.Mechanism(json.dumps(cut()), device=False).info
    assert inf.dense_block == 90 and inf.smem_per_cell_fp64 <= BLOCK


def _sections(mj, k):
    mj["aerosol"]["sections"] = k
    return mj


# gas mechanisms: blocks of 8..114 rows with every remainder by 4 and 8, on
# strides at and beyond the plain multiple; a block that starts late; split
# rows (64 lanes) and the water parameter's entries
MECHS = {f"gas{n}": (lambda n=n: gas(n)) for n in
         (10, 12, 24, 38, 40, 42, 44, 60, 76, 79, 80, 82, 84, 86, 100, 116, 117, 126, 141, 147)}
MECHS.update(cut=cut, water3=lambda: _sections(w.water_mechanism(), 3), multiphase8=w.multiphase_mechanism)


def _growth(M, perm):
    """|| |L| |U| ||_inf of the elimination in the order of `perm`."""
    A = M[np.ix_(perm, perm)].copy()
    n = len(A)
    for k in range(n - 1):
        A[k + 1:, k] /= A[k, k]
        A[k + 1:, k + 1:] -= np.outer(A[k + 1:, k], A[k, k + 1:])
    L, U = np.tril(A, -1) + np.eye(n), np.triu(A)
    return np.linalg.norm(np.abs(L) @ np.abs(U), np.inf)


@pytest.mark.gpu
@pytest.mark.parametrize("variant", [camp.VARIANT_FP64, camp.VARIANT_MIXED])
@pytest.mark.parametrize("name,lanes", [(k, l) for k in sorted(MECHS) for l in (32, 64)
                                        if (k, l) != ("cut", 64)])  # no room for partial sums
def test_lu_solve_backward_error(cuda, name, lanes, variant):
    """||M x - b|| within the bound of an elimination and two triangular
    solves, 3 n u || |L||U| || ||x||, with a factor of 4 for the rounding of
    J's entries (rate constant, up to two factors, coefficient, their sum) and
    of b."""
    import torch
    mj = MECHS[name]()
    gm, om = camp.Mechanism(json.dumps(mj)), oracle.Mechanism(json.dumps(mj))
    gm.set_lanes(lanes)
    y, env = w.cells(mj, 3, seed=7)
    b = np.random.default_rng(8).normal(size=y.shape)
    gamma = 0.1
    x, st = gm.lu_solve(torch.tensor(y, device=cuda), torch.tensor(env, device=cuda), gamma,
                        torch.tensor(b, device=cuda), variant=variant)
    x, st = x.cpu().numpy(), st.cpu().numpy()
    assert (st == 0).all()
    u = 2.0 ** -53 if variant == camp.VARIANT_FP64 else 2.0 ** -24
    perm = gm.structure()["perm"]
    for c in range(len(y)):
        kf, kr = om.rate_constants(env[c])
        M = np.eye(gm.n) - gamma * om.jacobian(kf, kr, y[c], env[c])
        bound = 12 * gm.n * u * _growth(M, perm) * np.abs(x[c]).max()
        assert np.abs(M @ x[c] - b[c]).max() <= bound
