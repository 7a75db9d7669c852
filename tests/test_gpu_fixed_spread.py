"""FP64 CG through the exact integer product (csrc/fixed.cuh) on matrices whose
diagonal spans nearly the 2^24 that it takes, and on the other side of the limit.

One shift serves the whole vector, so the small entries of an unpreconditioned
residual keep fewer bits than FP64 gives them.  The matrix is S A S with powers
of two in S, so that the exact iterates are known from extended precision.

Bar, per k iterations, relative to the iterate's 2-norm, in x and in S x:
4 k (27 + 4) 2^-53: in every iteration 27 products and sums of a row and four vector
operations, each of one rounding, with the sums of absolute values at most four times the
values'.  The shift's part stays below: scaled rows 2^12 apart at most leave an
entry of the small ones 2^-60 2^12 = 32 roundings."""
import numpy as np
import pytest

from paper_1107_0538_gb300 import gbcg, problems

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def scaled_box(edges, steps, graded):
    """S A S and S: S in powers of two over `steps` + 1 steps, in random rows or rising with the row."""
    g = problems.Grid(*edges, 1.0 / max(edges))
    A = problems.q1_matrix(problems.nu_blobs(g, nu_iron=1e-2), g.h)[0]
    e = np.arange(A.n) * (steps + 1) // A.n if graded else np.random.default_rng(7).integers(0, steps + 1, A.n)
    s = np.ldexp(1.0, e - steps // 2)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    return problems.CSR(A.n, A.rowptr, A.colidx, A.vals * s[rows] * s[A.colidx]), s


def iterate(A, b, k, jacobi):
    """CG's k-th iterate from 0 in extended precision."""
    T = np.longdouble
    cols, vals = np.zeros((A.n, 27), np.int64), np.zeros((A.n, 27), T)
    for j in range(27):
        has = np.diff(A.rowptr) > j
        at = A.rowptr[:-1][has] + j
        cols[has, j], vals[has, j] = A.colidx[at], A.vals[at]
    d = 1.0 / (vals * (cols == np.arange(A.n)[:, None])).sum(1) if jacobi else np.ones(A.n, T)
    x, r = np.zeros(A.n, T), b.astype(T)
    p = d * r
    rho = (r * p).sum()
    for _ in range(k):
        q = (vals * p[cols]).sum(1)
        a = rho / (p * q).sum()
        x, r = x + a * p, r - a * q
        new = (r * d * r).sum()
        p, rho = d * r + new / rho * p, new
    return x


# edges, grid_ctas, and the kernel with the integer and with the FP64 product
KERNELS = {"cluster": ((10, 9, 11), 0, "cg_cluster_kernel/int", "cg_sell_kernel/fp64"),
           "slices": ((10, 9, 11), 152, "cg_sell_kernel/int", "cg_sell_kernel/fp64"),
           "ring": ((13, 11, 9), 1, "cg_ring_kernel/int", "cg_sellmem_kernel/fp64")}


@pytest.mark.parametrize("jacobi", [0, 1])
@pytest.mark.parametrize("steps,graded", [(0, 0), (6, 0), (10, 1), (11, 1), (12, 1), (13, 0)],
                         ids=["2^7", "2^17", "2^22_graded", "2^24_graded", "2^26_graded", "2^29"])
@pytest.mark.parametrize("name", list(KERNELS))
def test_iterates_of_scaled_matrices(name, steps, graded, jacobi):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    edges, ctas, integer, fp64 = KERNELS[name]
    A, s = scaled_box(edges, steps, graded)
    d = A.vals[np.repeat(np.arange(A.n), np.diff(A.rowptr)) == A.colidx]
    b = problems.rhs_uniform(A.n, 3) * s
    c = np.frexp(d)[1] // 2   # the rows' exponents: 2^c is about the diagonal's root
    assert (c.max() - c.min() <= 12) == (steps <= 11)
    with gbcg.Solver(A, precond=jacobi, grid_ctas=ctas) as solver:
        assert solver.kernel() == (integer if steps <= 11 else fp64)
        for k in (1, 5):
            xt = torch.zeros(A.n, dtype=torch.float64, device="cuda:0")
            solver.solve(torch.from_numpy(b).to("cuda:0"), xt, tol=0.0, maxit=k)
            want, x = iterate(A, b, k, jacobi), xt.cpu().numpy()
            for w in (1.0, s):
                off, size = (x - want) * w, want * w
                assert np.sqrt((off * off).sum()) <= 4 * k * 31 * 2.0 ** -53 * np.sqrt((size * size).sum()), (k, w is s)
