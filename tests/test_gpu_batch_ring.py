"""Batched solves whose tiles are stored by their rows' common offsets
(csrc/batch.cu, batch_pass_ring) against the oracle's SpMV: ragged last tiles,
systems of one row and of many tiles per warp, rows at a system's edge whose
tile's offsets reach into the neighbouring system (which may hold NaN), and
batches that keep the staged tiles (more offsets than the limit, repeated
columns).  The solver stops on ||b - A x|| <= tol ||b|| in FP64; the same
residual recomputed here may differ by the rounding of one SpMV (5%)."""
import numpy as np
import pytest

import oracle
from paper_1107_0538_gb300 import gbcg, problems

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-8


def box(ex, ey, ez):
    g = problems.Grid(ex, ey, ez, 1.0 / max(ex, ey, ez))
    return problems.q1_matrix(problems.nu_blobs(g, nu_iron=1e-2), g.h, shift=1.0)[0]


def band(n, reach):
    """2 reach + 1 offsets in every inner row."""
    rowptr, cols, vals = [0], [], []
    for i in range(n):
        c = np.arange(max(0, i - reach), min(n, i + reach + 1))
        cols.append(c)
        vals.append(np.where(c == i, 2.0 * reach + 1.0, -1.0))
        rowptr.append(rowptr[-1] + len(c))
    return problems.CSR(n, np.array(rowptr, np.int32), np.concatenate(cols).astype(np.int32), np.concatenate(vals))


def with_repeats(A):
    """A with the diagonal of every third row stored as two halves."""
    rowptr, cols, vals = [0], [], []
    for i in range(A.n):
        c, v = A.colidx[A.rowptr[i]:A.rowptr[i + 1]], A.vals[A.rowptr[i]:A.rowptr[i + 1]].copy()
        if i % 3 == 0:
            v = np.where(c == i, 0.5 * v, v)
            c, v = np.append(c, i), np.append(v, v[c == i])
        cols.append(c)
        vals.append(v)
        rowptr.append(rowptr[-1] + len(c))
    return problems.CSR(A.n, np.array(rowptr, np.int32), np.concatenate(cols).astype(np.int32), np.concatenate(vals))


CASES = {
    "ragged": lambda: [box(5, 6, 7), band(1, 0), box(13, 11, 9), band(33, 2), box(4, 3, 2)],
    "many_tiles": lambda: [box(47, 44, 41), box(45, 47, 43), box(8, 8, 8)],  # tiles per warp > buffers
    "31_offsets": lambda: [band(3000, 15), box(9, 9, 9)],
    "33_offsets": lambda: [band(3000, 16), box(9, 9, 9)],
    "repeats": lambda: [with_repeats(box(9, 8, 7)), box(9, 9, 9)],
}


@pytest.mark.parametrize("values", [gbcg.CG_VALUES_FP32, gbcg.CG_VALUES_BF16], ids=["fp32", "bf16"])
@pytest.mark.parametrize("nan", [0, 1], ids=["", "nan_neighbour"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_batch_residuals(name, nan, values):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    mats = CASES[name]()
    rng = np.random.default_rng(3)
    at = np.concatenate([[0], np.cumsum([A.n for A in mats])])
    Bn = rng.standard_normal((4, at[-1]))
    if nan:   # the first system, last row: the next system's first rows are beside it
        Bn[1, at[1] - 1] = np.nan
    with gbcg.BatchSolver(mats, inner_values=values, precond=1) as bs:
        B = torch.from_numpy(Bn).to(dev)
        X = torch.zeros_like(B)
        _, res, _ = bs.solve(B, X, TOL)
    X = X.cpu().numpy()
    for s, A in enumerate(mats):
        for r in range(4):
            b, x = Bn[r, at[s]:at[s + 1]], X[r, at[s]:at[s + 1]]
            if nan and s == 0 and r == 1:
                assert res[s * 4 + r].status == gbcg.CG_ENAN
                continue
            assert res[s * 4 + r].status == gbcg.CG_OK, (s, r, res[s * 4 + r].status)
            assert np.linalg.norm(b - oracle.spmv(A, x)) <= 1.05 * TOL * np.linalg.norm(b), (s, r)
