"""Which kernel a handle's solves run (cg_kernel_name, cg_batch_kernel_name), on
both sides of the limits by which it is picked.  Every kernel falls back to
another correct one, so the tests that compare solutions would not notice a
kernel that is never picked; the matrices they use are named here with the
kernel they mean to reach."""
import numpy as np
import pytest

import oracle
import test_fixed
import test_gpu_batch_ring
import test_gpu_cluster
import test_gpu_ring
from paper_1107_0538_gb300 import gbcg, problems

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FP32, BF16 = dict(inner_values=gbcg.CG_VALUES_FP32), dict(inner_values=gbcg.CG_VALUES_BF16)
MEM = dict(vectors_in_memory=True)
fixed, ring, cluster, batch = test_fixed.CASES, test_gpu_ring.CASES, test_gpu_cluster.CASES, test_gpu_batch_ring.CASES


@pytest.fixture(scope="module", autouse=True)
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def box(ex, ey, ez):
    return test_gpu_ring.box(ex, ey, ez)


def scaled_rows(spread):
    """Band matrix whose diagonal spans a factor of spread (a power of two), in two steps."""
    A = test_fixed.banded(600, 7, 8)
    s = np.where(np.arange(A.n) < 300, 1.0, spread ** 0.5)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    d = A.to_dense().diagonal()
    v = A.vals / np.sqrt(d[rows] * d[A.colidx]) * 1.5   # diagonal 1.5: its exponent is away from a rounding edge
    return problems.CSR(A.n, A.rowptr, A.colidx, v * s[rows] * s[A.colidx])


def row_sum(total):
    """Diagonal 1 and 30 equal off-diagonals in the inner rows, |row| summing to total there."""
    A = test_fixed.banded(600, 31, 9)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    return problems.CSR(A.n, A.rowptr, A.colidx, np.where(rows == A.colidx, 1.0, -(total - 1.0) / 30.0))


def negative_diagonal():
    A = test_fixed.banded(600, 7, 8)
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    return problems.CSR(A.n, A.rowptr, A.colidx, np.where((rows == 17) & (A.colidx == 17), -A.vals, A.vals))


def points(*dims):
    """Weighted Laplacian of a grid (5 or 7 points), shifted."""
    idx = np.arange(int(np.prod(dims))).reshape(dims)
    i, j = [], []
    for ax in range(len(dims)):
        a = np.moveaxis(idx, ax, 0)
        i.append(a[:-1].ravel())
        j.append(a[1:].ravel())
    i, j = np.concatenate(i), np.concatenate(j)
    w = np.random.default_rng(1).uniform(0.5, 1.0, i.size)
    n = idx.size
    d = 1e-2 + np.bincount(i, w, n) + np.bincount(j, w, n)
    key = np.concatenate([i * n + j, j * n + i, np.arange(n) * (n + 1)])
    order = np.argsort(key)
    rowptr = np.searchsorted(key[order], np.arange(n + 1, dtype=np.int64) * n).astype(np.int32)
    return problems.CSR(n, rowptr, (key[order] % n).astype(np.int32), np.concatenate([-w, -w, d])[order])


def with_hub(A, m):
    """A with row 777 coupled to m further rows, spread over the matrix, weakly enough to stay definite."""
    rows = np.repeat(np.arange(A.n), np.diff(A.rowptr))
    others = np.setdiff1d(np.linspace(0, A.n - 1, m + 40).astype(int), A.colidx[A.rowptr[777]:A.rowptr[778]])[:m]
    w = np.full(m, 1e-9)
    hub = np.full(m, 777)
    key = np.concatenate([rows.astype(np.int64) * A.n + A.colidx, hub * A.n + others, others * A.n + hub])
    order = np.argsort(key, kind="stable")
    key = key[order]
    assert np.all(np.diff(key) > 0)
    rowptr = np.searchsorted(key, np.arange(A.n + 1, dtype=np.int64) * A.n).astype(np.int32)
    return problems.CSR(A.n, rowptr, (key % A.n).astype(np.int32), np.concatenate([A.vals, w, w])[order])


# name: (matrix, options, kernel)
CASES = {
    # one cluster, the slices of the grid, the ring, by size
    "box8": (lambda: box(8, 8, 8), {}, "cg_cluster_kernel/int"),
    "box8_jacobi": (lambda: box(8, 8, 8), dict(precond=1), "cg_cluster_kernel/int"),
    "box20": (lambda: box(20, 20, 20), {}, "cg_cluster_kernel/int"),
    "box24": (cluster["24cube"], {}, "cg_sell_kernel/int"),
    "box50": (lambda: box(50, 50, 50), {}, "cg_sell_kernel/int"),
    "chip": (ring["chip"][0], {}, "cg_ring_kernel/int"),
    "box60": (lambda: box(60, 60, 60), dict(precond=1), "cg_ring_kernel/int"),
    # windows of a cluster's CTAs that fit, and that do not
    "513_rows": (cluster["17_slices"], {}, "cg_cluster_kernel/int"),
    "flat": (cluster["flat_box"], {}, "cg_cluster_kernel/int"),
    # a given CTA count asks for the grid
    "box8_grid": (lambda: box(8, 8, 8), dict(grid_ctas=152), "cg_sell_kernel/int"),
    "5point": (lambda: points(90, 90), dict(grid_ctas=4), "cg_ring_kernel/int"),
    "5point_jacobi": (lambda: points(90, 90), dict(grid_ctas=4, precond=1), "cg_sellmem_kernel/fp64"),
    "7point_jacobi": (lambda: points(20, 20, 20), dict(grid_ctas=4, precond=1), "cg_ring_kernel/int"),
    "two_ctas": (ring["two_ctas"][0], dict(grid_ctas=2), "cg_ring_kernel/int"),
    "one_cta": (ring["one_cta"][0], dict(grid_ctas=1), "cg_ring_kernel/int"),
    "ten_ctas": (lambda: box(20, 20, 20), dict(grid_ctas=10), "cg_sell_kernel/int"),
    # short rows: integers only where they make the cluster possible
    "7point20": (lambda: points(20, 20, 20), {}, "cg_cluster_kernel/int"),
    "7point40": (lambda: points(40, 40, 40), {}, "cg_sell_kernel/fp64"),
    "7point38": (lambda: points(38, 38, 38), {}, "cg_sell_kernel/int"),     # 361 rows per CTA
    "width7": (lambda: test_fixed.banded(3000, 7, 1), dict(grid_ctas=4), "cg_sell_kernel/fp64"),
    "width7_8_ctas": (lambda: test_fixed.banded(3000, 7, 1), dict(grid_ctas=8), "cg_sell_kernel/int"),
    "width9": (lambda: test_fixed.banded(3000, 9, 1), dict(grid_ctas=4), "cg_sell_kernel/int"),
    "width9_jacobi": (lambda: test_fixed.banded(3000, 9, 1), dict(grid_ctas=4, precond=1), "cg_sell_kernel/fp64"),
    "width11_jacobi": (lambda: test_fixed.banded(3000, 11, 1), dict(grid_ctas=4, precond=1), "cg_sell_kernel/int"),
    # limits of the integer product
    "width31": (fixed["width31"][0], dict(grid_ctas=152), "cg_sell_kernel/int"),
    "width33": (fixed["width33"][0], dict(grid_ctas=152), "cg_sell_kernel/fp64"),
    "width33_ring": (fixed["width33"][0], dict(grid_ctas=1), "cg_sellmem_kernel/fp64"),
    "far32767": (fixed["far32767"][0], {}, "cg_sell_kernel/int"),
    "far32768": (fixed["far32768"][0], {}, "cg_sell_kernel/fp64"),
    "scaled": (fixed["scaled"][0], dict(grid_ctas=152), "cg_sell_kernel/int"),
    "scaled_wide": (fixed["scaled_wide"][0], dict(grid_ctas=152), "cg_sell_kernel/fp64"),
    "spread24": (lambda: scaled_rows(2.0 ** 24), dict(grid_ctas=152), "cg_sell_kernel/int"),
    "spread26": (lambda: scaled_rows(2.0 ** 26), dict(grid_ctas=152), "cg_sell_kernel/fp64"),
    "sum63.9": (lambda: row_sum(63.9), dict(grid_ctas=152), "cg_sell_kernel/int"),
    "sum64.1": (lambda: row_sum(64.1), dict(grid_ctas=152), "cg_sell_kernel/fp64"),
    "negative": (negative_diagonal, {}, "cg_sell_kernel/fp64"),
    # repeated columns and too many offsets leave the ring
    "repeats": (ring["repeats"][0], dict(grid_ctas=2), "cg_sellmem_kernel/fp64"),
    "memory": (lambda: box(8, 8, 8), MEM, "cg_solve_kernel/fp64"),
    # a long row, which one warp of a SELL-32 slice would walk alone
    "mid_hub120": (lambda: with_hub(box(53, 54, 55), 102), {}, "cg_sellmem_kernel/fp64"),
    "mid_hub121": (lambda: with_hub(box(53, 54, 55), 103), {}, "cg_solve_kernel/fp64"),
    "mid_hub2000": (lambda: with_hub(box(53, 54, 55), 2000), dict(precond=1), "cg_solve_kernel/fp64"),
    "large_hub2000": (lambda: with_hub(box(20, 20, 20), 2000), dict(grid_ctas=1), "cg_sellmem_kernel/fp64"),
    # refinement
    "fp32": (lambda: box(8, 8, 8), FP32, "cg_irring_kernel"),
    "bf16": (lambda: box(8, 8, 8), dict(precond=1, **BF16), "cg_irring_kernel"),
    "fp32_mid": (ring["chip"][0], FP32, "cg_irring_kernel"),
    "fp32_repeats": (lambda: test_gpu_ring.with_repeats(box(8, 8, 8)), FP32, "cg_irsell_kernel"),
    "bf16_width33": (fixed["width33"][0], BF16, "cg_irsell_kernel"),
    "fp32_repeats_two_ctas": (ring["repeats"][0], dict(grid_ctas=2, **FP32), "cg_ir_kernel"),
    "fp32_memory": (lambda: box(8, 8, 8), dict(**FP32, **MEM), "cg_ir_kernel"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_solve_kernel(name):
    make, kw, want = CASES[name]
    with gbcg.Solver(make(), **kw) as s:
        assert s.kernel() == want


@pytest.mark.parametrize("precond", [0, 1])
@pytest.mark.parametrize("edges,ctas", [((53, 54, 55), 0), ((20, 20, 20), 6), ((9, 9, 30), 3)],
                         ids=["chip", "six_ctas", "three_ctas"])
def test_long_row_iterates(dev, edges, ctas, precond):
    """The tiled kernel with a thread's rows in registers, one row of 800 entries: 1e-10 from the oracle at a fixed iteration count, the bar of the
    FP64 kernels, and a full solve's own and true residual."""
    A = with_hub(box(*edges), 800)
    b = problems.rhs_uniform(A.n, 31)
    with gbcg.Solver(A, precond=precond, grid_ctas=ctas) as s:
        assert s.kernel() == "cg_solve_kernel/fp64" and s.plan()["reg_rows"] > 0
        for k in (1, 2, 40):
            ref = oracle.cg(A, b, tol=0.0, maxit=k, precond=precond)
            xt = torch.zeros(A.n, dtype=torch.float64, device=dev)
            info = s.solve(torch.from_numpy(b).to(dev), xt, tol=0.0, maxit=k)
            assert info.iters == k and np.linalg.norm(xt.cpu().numpy() - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])
        xt.zero_()
        info = s.solve(torch.from_numpy(b).to(dev), xt, tol=1e-9)
        true = np.linalg.norm(b - oracle.spmv(A, xt.cpu().numpy())) / np.linalg.norm(b)
        assert info.status == gbcg.CG_OK and info.relres <= 1e-9 and true <= 1.05e-9


@pytest.mark.parametrize("name,want", [("ragged", "offsets"), ("many_tiles", "offsets"), ("31_offsets", "offsets"),
                                       ("33_offsets", "staged"), ("repeats", "staged")])
@pytest.mark.parametrize("values", [gbcg.CG_VALUES_FP32, gbcg.CG_VALUES_BF16], ids=["fp32", "bf16"])
def test_batch_kernel(name, want, values):
    with gbcg.BatchSolver(batch[name](), inner_values=values, precond=1) as bs:
        assert bs.kernel() == "cg_batch_kernel/" + want
        for gather, lanes, static in ((1, 1, 0), (0, 2, 0), (0, 4, 1)):
            bs.set_tuning(1e-3, gather, lanes, static)
            assert bs.kernel() == "cg_batch_kernel/staged"
        bs.set_tuning(1e-3, 0, 1, 1)
        assert bs.kernel() == "cg_batch_kernel/" + want


def test_learned_kernel():
    inst = problems.learn_instance(8, 20001)
    net = gbcg.Net(problems.learn_init_params())
    for kw, want in (({}, "fcg_sell_kernel"), (MEM, "fcg_spmv_kernel")):
        with gbcg.Solver(inst.A, precond=gbcg.CG_PRECOND_LEARNED, **kw) as s:
            assert s.kernel() == ""
            s.set_learned(net, inst.grid, inst.lognu.astype(np.float32))
            assert s.kernel() == want
    net.close()


def test_no_handle():
    assert gbcg.cg_kernel_name(None) == "" and gbcg.cg_batch_kernel_name(None) == ""
