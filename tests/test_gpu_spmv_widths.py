"""Stand-alone SpMV on bands of every width around its batch size (the rest of a
slice of width w is one batch of w mod 9 entries), with 16-bit and 32-bit
columns.  Bar per row: two summation orders of m products, 2 (m + 2) 2^-53
sum |a x|."""
import numpy as np
import pytest

import oracle
from paper_1107_0538_gb300 import gbcg, problems

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def band(n, width, far):
    """`width` entries a row: the columns from the row on (round the end), the last one `far` rows on."""
    offs = np.arange(width)
    if width > 1 and far:
        offs[-1] = far
    cols = np.sort((np.arange(n)[:, None] + offs) % n, axis=1)
    vals = np.random.default_rng(width).standard_normal((n, width))
    return problems.CSR(n, np.arange(0, n * width + 1, width, dtype=np.int32), cols.astype(np.int32).ravel(), vals.ravel())


@pytest.mark.parametrize("n,far", [(1000, 0), (70001, 35000)], ids=["16bit", "32bit"])
@pytest.mark.parametrize("width", list(range(1, 20)) + [27, 28, 35])
def test_band_widths(n, far, width):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A = band(n, width, far)
    x = np.random.default_rng(3).standard_normal(n)
    with gbcg.Solver(A, vectors_in_memory=True) as s:
        xt = torch.from_numpy(x).to("cuda:0")
        yt = torch.full_like(xt, float("nan"))
        s.spmv(xt, yt)
        y = yt.cpu().numpy()
    absum = np.abs(A.vals.reshape(n, width) * x[A.colidx.reshape(n, width)]).sum(1)
    assert np.all(np.abs(y - oracle.spmv(A, x)) <= 2.0 * (width + 2) * 2.0 ** -53 * absum)
