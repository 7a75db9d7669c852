"""The exact integer product of the FP64 solve kernels (csrc/fixed.cuh).

On the CPU: its conversions and limb sums against exact 128-bit integers.  On
the GPU: solves through it against the oracle at a fixed iteration count, at
the edges of the matrices it takes (row widths, column offsets, diagonals) and
beyond them, where the FP64 product answers.
"""
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1107_0538_gb300 import gbcg, problems
from paper_1107_0538_gb300.build import nvcc_path

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_integer_arithmetic_against_128_bits(tmp_path):
    if os.uname().machine != "x86_64":
        pytest.skip("compares with the 64-bit mantissa of x87 long double")
    exe = tmp_path / "fixed_check"
    subprocess.run([nvcc_path(), "-O1", "-std=c++17", "-gencode=arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "paper_1107_0538_gb300", "csrc"), "-o", str(exe),
                    os.path.join(ROOT, "tests", "fixed_check.cu")], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, f"{res.stdout.strip()} mismatches"


def banded(n, width, seed, spread=1.0, far=0):
    """Symmetric positive definite band matrix: `width` entries in the middle
    rows (columns i - (width-1)/2 .. ), rows and columns scaled by factors in
    [1/spread, spread]; far > 0 moves the outermost pair `far` columns away."""
    rng = np.random.default_rng(seed)
    half = (width - 1) // 2
    offs = list(range(1, half + 1))
    if far:
        offs[-1] = far
    M = {}
    for o in offs:
        v = -rng.uniform(0.1, 1.0, max(n - o, 0))
        for i in range(n - o):
            M[(i, i + o)] = M[(i + o, i)] = v[i]
    d = np.full(n, 1e-2)
    for (i, _), v in M.items():
        d[i] -= v
    s = spread ** rng.uniform(-1.0, 1.0, n)
    rows = [[] for _ in range(n)]
    for (i, j), v in M.items():
        rows[i].append((j, v * s[i] * s[j]))
    rowptr, cols, vals = [0], [], []
    for i in range(n):
        r = sorted(rows[i] + [(i, d[i] * s[i] * s[i])])
        cols += [c for c, _ in r]
        vals += [v for _, v in r]
        rowptr.append(len(cols))
    return problems.CSR(n, np.array(rowptr, np.int32), np.array(cols, np.int32), np.array(vals))


# (matrix, iterations): 31 entries a row are the most the integers take, 33 go
# to the FP64 product, as does a column more than 32767 rows away; one row, a
# last slice of one row, a diagonal spread over 10^6 (integers) and 10^12 (FP64)
CASES = {
    "width31": (lambda: banded(2000, 31, 1), 25),
    "width33": (lambda: banded(2000, 33, 2), 25),
    "tail1": (lambda: banded(993, 9, 3), 25),
    "tail31": (lambda: banded(1023, 5, 4), 25),
    "scaled": (lambda: banded(1500, 11, 5, spread=30.0), 25),
    "scaled_wide": (lambda: banded(1500, 11, 5, spread=1e3), 8),
    "far32767": (lambda: banded(34000, 5, 6, far=32767), 25),
    "far32768": (lambda: banded(34000, 5, 7, far=32768), 25),
    "uneven_box": (lambda: problems.q1_matrix(problems.nu_blobs(problems.Grid(13, 29, 7, 0.05)), 0.05)[0], 40),
    "two_slices_a_warp": (lambda: problems.q1_matrix(problems.nu_blobs(problems.Grid(57, 53, 51, 0.02)), 0.02)[0], 40),
}


def solve(A, b, tol, maxit, precond, dev, **kw):
    import torch
    with gbcg.Solver(A, precond=precond, **kw) as s:
        bt = torch.from_numpy(np.ascontiguousarray(b)).to(dev)
        xt = torch.zeros_like(bt)
        info = s.solve(bt, xt, tol=tol, maxit=maxit)
        return xt.cpu().numpy(), info


@pytest.fixture(scope="module")
def dev():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.gpu
# the scaled systems with Jacobi only: without it their 25 iterations amplify
# rounding until two CPU FP64 codes differ by 4e-10
@pytest.mark.parametrize("name,precond", [(n, p) for n in CASES for p in (0, 1) if p or not n.startswith("scaled")])
def test_iterates_match_oracle(dev, name, precond):
    """Relative difference at most 1e-10 at a fixed iteration count, the bar of
    the other FP64 kernels; both products stay far inside it."""
    make, k = CASES[name]
    A = make()
    b = problems.rhs_uniform(A.n, 3)
    if name.startswith("scaled"):
        b = b * np.sqrt(A.to_dense().diagonal())
    ref = oracle.cg(A, b, tol=0.0, maxit=k, precond=precond)
    x, info = solve(A, b, 0.0, k, precond, dev)
    assert info.iters == k == ref["iters"] and info.status == gbcg.CG_ENOCONV
    assert np.linalg.norm(x - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])


@pytest.mark.gpu
@pytest.mark.parametrize("precond", [0, 1])
@pytest.mark.parametrize("sa,sb", [(40, 0), (-40, 60), (0, -120), (-30, 30)])
def test_powers_of_two_scale_the_solution_exactly(dev, sa, sb, precond):
    """A and b times powers of two change no rounding (A's an even power: its
    diagonal's roots are powers of two then), so x scales bit for bit."""
    pr = problems.cube_blobs(9, contrast=1e3)
    x, i0 = solve(pr.A, pr.b, 1e-10, 0, precond, dev)
    A = problems.CSR(pr.A.n, pr.A.rowptr, pr.A.colidx, np.ldexp(pr.A.vals, sa))
    y, i1 = solve(A, np.ldexp(pr.b, sb), 1e-10, 0, precond, dev)
    assert i0.status == i1.status == gbcg.CG_OK and i0.iters == i1.iters
    assert np.array_equal(np.ldexp(x, sb - sa), y)


@pytest.mark.gpu
def test_infinite_and_nan_entries_keep_their_status(dev):
    """A matrix with an entry that is not finite goes to the FP64 product;
    right-hand sides that are not finite, or overflow, end in CG_ENAN."""
    pr = problems.cube_blobs(6)
    for v in (np.inf, np.nan):
        A = problems.CSR(pr.A.n, pr.A.rowptr, pr.A.colidx, pr.A.vals.copy())
        A.vals[17] = v
        assert solve(A, pr.b, 1e-8, 0, 0, dev)[1].status == gbcg.CG_ENAN
        b = pr.b.copy()
        b[3] = v
        assert solve(pr.A, b, 1e-8, 0, 0, dev)[1].status == gbcg.CG_ENAN
    assert solve(pr.A, pr.b * 1e200, 1e-8, 0, 0, dev)[1].status == gbcg.CG_ENAN
