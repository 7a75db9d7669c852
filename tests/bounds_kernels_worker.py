"""Runs every solve kernel of the bounds-check build, by name (cg_kernel_name,
cg_batch_kernel_name), and prints one JSON line: what ran, how each solve ended,
and the index faults counted.  GBCG_LIBRARY=check must be set by the caller.
Helper of test_gpu_bounds_kernels.py."""
import json
import os
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, os.path.dirname(HERE))
sys.path.insert(0, HERE)

import numpy as np  # noqa: E402
import torch  # noqa: E402

import oracle  # noqa: E402
import test_fixed  # noqa: E402
import test_gpu_batch_ring  # noqa: E402
import test_gpu_kernel_choice  # noqa: E402
import test_gpu_ring  # noqa: E402
from paper_1107_0538_gb300 import gbcg, problems  # noqa: E402

assert gbcg.LIB_PATH.endswith("libgbcg_check.so"), gbcg.LIB_PATH
dev = torch.device("cuda:0")
FP32, BF16 = dict(inner_values=gbcg.CG_VALUES_FP32), dict(inner_values=gbcg.CG_VALUES_BF16)
box = test_gpu_ring.box
thin = box(5, 31, 40)                                # a last slice of 15 rows
cubes, band33 = box(20, 20, 20), test_fixed.CASES["width33"][0]()
repeats = test_gpu_ring.with_repeats(box(9, 8, 7))
repeats_mid = test_gpu_ring.with_repeats(box(17, 18, 19))
hub = test_gpu_kernel_choice.with_hub(box(9, 9, 30), 800)

SOLVES = [
    (box(8, 8, 8), {}), (thin, dict(precond=1)),                                    # cluster
    (thin, dict(grid_ctas=152)), (cubes, dict(grid_ctas=10, precond=1)),            # slices, integers
    (band33, dict(grid_ctas=152)), (repeats, dict(vectors_in_memory=True)),
    (cubes, dict(grid_ctas=2)), (thin, dict(grid_ctas=1, precond=1)),               # ring
    (repeats_mid, dict(grid_ctas=2)), (band33, dict(grid_ctas=1, precond=1)),       # SELL-32 in memory
    (hub, dict(grid_ctas=3)), (hub, dict(grid_ctas=3, precond=1)),                  # tiles, rows in registers
    (thin, FP32), (thin, dict(grid_ctas=1, precond=1, **BF16)), (cubes, dict(grid_ctas=2, **FP32)),
    (repeats, FP32), (band33, dict(precond=1, **BF16)),                             # refinement on slices
    (repeats_mid, dict(grid_ctas=2, **FP32)), (thin, dict(vectors_in_memory=True, **BF16)),
]
out = {"solves": [], "batch": []}
for A, kw in SOLVES:
    b = problems.rhs_uniform(A.n, 41)
    with gbcg.Solver(A, **kw) as s:
        x = torch.zeros(A.n, dtype=torch.float64, device=dev)
        info = s.solve(torch.from_numpy(b).to(dev), x, tol=1e-8)
        true = float(np.linalg.norm(b - oracle.spmv(A, x.cpu().numpy())) / np.linalg.norm(b))
        out["solves"].append({"kernel": s.kernel(), "n": A.n, "kw": str(kw), "status": info.status, "relres_true": true})
for name in ("ragged", "31_offsets", "33_offsets"):
    mats = test_gpu_batch_ring.CASES[name]()
    for values in (gbcg.CG_VALUES_FP32, gbcg.CG_VALUES_BF16):
        for tuning in (None, (1e-3, 0, 1, 1), (1e-3, 1, 1, 0), (1e-3, 0, 2, 0)):
            with gbcg.BatchSolver(mats, inner_values=values, precond=1) as bs:
                if tuning:
                    bs.set_tuning(*tuning)
                B = torch.from_numpy(np.random.default_rng(3).standard_normal((3, bs.n))).to(dev)
                X = torch.zeros_like(B)
                rc, res, _ = bs.solve(B, X, 1e-8)
                out["batch"].append({"kernel": bs.kernel(), "name": name, "tuning": tuning, "status": rc})
torch.cuda.synchronize()
out["faults"] = gbcg.cg_bounds_faults()
print(json.dumps(out))
