"""Solves whose matrix runs through the shared-memory ring (csrc/ring.cuh)
against the oracle: a CTA with more slices than warps, with fewer and with more
slots than slices, ragged ends, slices of several widths, and matrices the ring
refuses (too many offsets, repeated columns), which other kernels solve."""
import numpy as np
import pytest

import oracle
from paper_1107_0538_gb300 import gbcg, problems

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def box(ex, ey, ez, contrast=1e2):
    g = problems.Grid(ex, ey, ez, 1.0 / max(ex, ey, ez))
    return problems.q1_matrix(problems.nu_blobs(g, nu_iron=1.0 / contrast), g.h)[0]


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


# matrix, grid_ctas: on few CTAs a small box has more slices per CTA than the
# slice kernel takes (31) and than the ring has slots
CASES = {
    "one_cta": (lambda: box(13, 11, 9), 1),        # 53 slices, 23 fixed-point slots
    "two_ctas": (lambda: box(20, 20, 20), 2),      # 145 slices each
    "seven_ctas": (lambda: box(31, 17, 23), 7),    # uneven ranges, a last slice of 16 rows
    "flat": (lambda: box(63, 60, 1), 3),           # 18 offsets a row, 12 and 8 at the edges
    "chip": (lambda: box(53, 54, 55), 0),
    "repeats": (lambda: with_repeats(box(20, 20, 20)), 2),
}


def solve(A, b, tol, maxit, dev, **kw):
    with gbcg.Solver(A, **kw) as s:
        xt = torch.zeros(A.n, dtype=torch.float64, device=dev)
        info = s.solve(torch.from_numpy(b).to(dev), xt, tol=tol, maxit=maxit)
        return xt.cpu().numpy(), info


@pytest.mark.parametrize("precond", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_fp64_iterates_match_oracle(dev, name, precond):
    """1e-10 at a fixed iteration count, the bar of the FP64 kernels, and a full
    solve's own and true residual."""
    make, ctas = CASES[name]
    A = make()
    b = problems.rhs_uniform(A.n, 21)
    for k in (1, 2, 30):
        ref = oracle.cg(A, b, tol=0.0, maxit=k, precond=precond)
        x, info = solve(A, b, 0.0, k, dev, precond=precond, grid_ctas=ctas)
        assert info.iters == k and info.status == gbcg.CG_ENOCONV
        assert np.linalg.norm(x - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])
    x, info = solve(A, b, 1e-9, 0, dev, precond=precond, grid_ctas=ctas)
    true = np.linalg.norm(b - oracle.spmv(A, x)) / np.linalg.norm(b)
    assert info.status == gbcg.CG_OK and info.relres <= 1e-9 and true <= 1.05e-9


@pytest.mark.parametrize("values", [gbcg.CG_VALUES_FP32, gbcg.CG_VALUES_BF16], ids=["fp32", "bf16"])
@pytest.mark.parametrize("name", list(CASES))
def test_refinement_and_inner_product(dev, name, values):
    """Refinement to 1e-9 of the true residual; y = A_lo x row by row within the
    bound of two FP32 summation orders."""
    make, ctas = CASES[name]
    A = make()
    b = problems.rhs_uniform(A.n, 22)
    for precond in (0, 1):
        x, info = solve(A, b, 1e-9, 0, dev, precond=precond, grid_ctas=ctas, inner_values=values)
        true = np.linalg.norm(b - oracle.spmv(A, x)) / np.linalg.norm(b)
        assert info.status == gbcg.CG_OK and true <= 1.0001e-9
    fmt = oracle.FP32_FORMAT if values == gbcg.CG_VALUES_FP32 else oracle.BF16_FORMAT
    if name == "repeats":
        return   # the two halves of a diagonal are off-diagonals to no one
    lo = problems.CSR(A.n, A.rowptr, A.colidx, oracle.lowprec_values(A, fmt))
    xs = problems.rhs_uniform(A.n, 23).astype(np.float32)
    with gbcg.Solver(A, grid_ctas=ctas, inner_values=values) as s:
        yt = torch.full((A.n,), float("nan"), dtype=torch.float32, device=dev)
        s.spmv_inner(torch.from_numpy(xs).to(dev), yt)
        y = yt.cpu().numpy().astype(np.float64)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    absum = np.bincount(rows, weights=np.abs(lo.vals * xs[A.colidx].astype(np.float64)), minlength=A.n)
    m = np.diff(A.rowptr)
    assert np.all(np.abs(y - oracle.spmv(lo, xs.astype(np.float64))) <= 2.0 * (m + 2) * (2.0 ** -24 + 2.0 ** -53) * absum)


def test_timeout_and_next_solve(dev):
    A = box(20, 20, 20)
    b = problems.rhs_uniform(A.n, 24)
    for values in (gbcg.CG_VALUES_FP64, gbcg.CG_VALUES_FP32):
        kw = dict(grid_ctas=2, inner_values=values)
        assert solve(A, b, 1e-9, 0, dev, wait_limit_s=2e-3, debug_phantom_arrivals=1, **kw)[1].status == gbcg.CG_ETIMEOUT
        assert solve(A, b, 1e-9, 0, dev, **kw)[1].status == gbcg.CG_OK


def test_two_handles_of_different_ring_sizes(dev):
    """Solves on one handle while another with larger slots exists."""
    A, B = box(20, 20, 20), box(63, 60, 1)
    with gbcg.Solver(A, grid_ctas=2) as sa, gbcg.Solver(B, grid_ctas=1) as sb:
        for s, M in ((sa, A), (sb, B), (sa, A)):
            b = problems.rhs_uniform(M.n, 25)
            xt = torch.zeros(M.n, dtype=torch.float64, device=dev)
            info = s.solve(torch.from_numpy(b).to(dev), xt, tol=1e-9)
            assert info.status == gbcg.CG_OK
            assert np.linalg.norm(b - oracle.spmv(M, xt.cpu().numpy())) <= 1.05e-9 * np.linalg.norm(b)
