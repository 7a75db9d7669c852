"""How far cg_solve_noalloc's iterates are from those of exact arithmetic.

CG in FP64 with q = A p formed anew in every iteration keeps its iterates near
the exact ones; a q that is carried along (q = A r + beta q) collects the
rounding of every iteration before.  The distance to iterates in extended
precision is compared with that of the textbook recurrence in FP64 (numpy) on
the same systems.  Two FP64 codes that only add in another order scatter by a
factor of e^0.25 per system, so the geometric mean over six systems lies in
1 +- 0.3 for a textbook code; a carried q gives 4 to 5.
"""
import math

import numpy as np
import pytest

from paper_1107_0538_gb300 import gbcg, problems

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

K = 60


def ell(A, T):
    """Columns and values of A, 27 per row (zeros at column 0 beyond a row's end)."""
    w = int(np.diff(A.rowptr).max())
    cols, vals = np.zeros((A.n, w), np.int64), np.zeros((A.n, w), T)
    for k in range(w):
        has = np.diff(A.rowptr) > k
        at = A.rowptr[:-1][has] + k
        cols[has, k], vals[has, k] = A.colidx[at], A.vals[at]
    return cols, vals


def textbook(A, b, T):
    cols, vals = ell(A, T)
    x, r = np.zeros(A.n, T), b.astype(T)
    p, rho = r.copy(), (r * r).sum()
    for _ in range(K):
        q = (vals * p[cols]).sum(1)
        a = rho / (p * q).sum()
        x, r = x + a * p, r - a * q
        new = (r * r).sum()
        p, rho = r + new / rho * p, new
    return x


def test_error_is_that_of_the_textbook_recurrence():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    ratios = []
    for e in (20, 22, 24):
        g = problems.Grid(e, e + 1, e - 2, 1.0 / e)
        A = problems.q1_matrix(problems.nu_blobs(g, nu_iron=1e-3), g.h)[0]
        keep = [torch.from_numpy(v).to(dev) for v in (A.rowptr, A.colidx, A.vals)]
        csr = gbcg.cg_csr(A.n, A.nnz, *(t.data_ptr() for t in keep), gbcg.CG_MEM_DEVICE)
        for seed in (3, 4):
            b = problems.rhs_uniform(A.n, seed)
            bt = torch.from_numpy(b).to(dev)
            xt = torch.zeros_like(bt)
            rc, info = gbcg.cg_solve_noalloc(csr, bt.data_ptr(), xt.data_ptr(), 0.0, K, None)
            assert rc == gbcg.CG_ENOCONV and info.iters == K
            exact = textbook(A, b, np.longdouble)

            def off(x):
                return float(np.linalg.norm((x - exact).astype(np.float64)))
            ratios.append(off(xt.cpu().numpy()) / off(textbook(A, b, np.float64)))
    assert math.exp(np.mean(np.log(ratios))) <= 2.0, ratios
