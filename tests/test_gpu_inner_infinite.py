"""y = A_lo x (cg_spmv_inner) with infinite and NaN entries in x: only the rows
that hold such a column take part.  In the slices with common offsets a row
also stores zeros at offsets it does not have; those add nothing."""
import numpy as np
import pytest

import oracle
from inner_bounds import lowprec_matrix, spmv_row_bound
from paper_1107_0538_gb300 import gbcg, problems

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
FORMATS = {gbcg.CG_VALUES_FP32: oracle.FP32_FORMAT, gbcg.CG_VALUES_BF16: oracle.BF16_FORMAT}


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("ctas", [0, 1], ids=["resident", "streamed"])
@pytest.mark.parametrize("values", list(FORMATS), ids=["fp32", "bf16"])
def test_other_rows_stay_finite(values, ctas, bad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = problems.Grid(13, 11, 9, 1.0 / 13)
    A = problems.q1_matrix(problems.nu_blobs(g, nu_iron=1e-2), g.h)[0]
    A.vals[A.rowptr[700] + 3] = 0.0   # a stored zero, in a row and column of finite x
    lo = lowprec_matrix(A, FORMATS[values])
    x = problems.rhs_uniform(A.n, 5).astype(np.float32).astype(np.float64)
    at = np.array([0, 13, 14, 400, 1007, A.n - 1])   # ends of lines, faces, the corners
    finite = x.copy()
    x[at] = bad
    with gbcg.Solver(A, inner_values=values, grid_ctas=ctas) as s:
        assert s.kernel() == "cg_irring_kernel"
        yt = torch.zeros(A.n, dtype=torch.float32, device="cuda:0")
        s.spmv_inner(torch.from_numpy(x.astype(np.float32)).to("cuda:0"), yt)
        y = yt.cpu().numpy().astype(np.float64)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    touched = np.zeros(A.n, bool)
    touched[rows[np.isin(A.colidx, at)]] = True
    assert not np.isfinite(y[touched]).any()
    err = np.abs(y - oracle.spmv(lo, finite))[~touched]
    assert np.all(err <= spmv_row_bound(lo, finite)[~touched])
