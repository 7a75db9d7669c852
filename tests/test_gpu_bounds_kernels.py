"""Every solve kernel in the bounds-check build, on ragged and small systems:
the kernels that the cluster and the ring replaced as the default choice for
such systems too.  On well-formed inputs no index fault is counted; solves meet
the tolerance in the residual recomputed on the CPU (5% for its rounding)."""
import json
import os
import subprocess
import sys

import pytest

from paper_1107_0538_gb300 import build as nvbuild
from paper_1107_0538_gb300 import gbcg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_every_kernel_counts_no_fault():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvbuild.build()
    res = subprocess.run([sys.executable, os.path.join(HERE, "bounds_kernels_worker.py")],
                         env=dict(os.environ, GBCG_LIBRARY="check"), capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stderr[-3000:]
    out = json.loads(res.stdout.strip().splitlines()[-1])
    assert out["faults"] == 0, out
    assert {s["kernel"] for s in out["solves"]} == {
        "cg_cluster_kernel/int", "cg_sell_kernel/int", "cg_sell_kernel/fp64", "cg_ring_kernel/int",
        "cg_sellmem_kernel/fp64", "cg_solve_kernel/fp64", "cg_irring_kernel", "cg_irsell_kernel", "cg_ir_kernel"}
    for s in out["solves"]:
        assert s["status"] == gbcg.CG_OK and s["relres_true"] <= 1.05e-8, s
    assert {b["kernel"] for b in out["batch"]} == {"cg_batch_kernel/offsets", "cg_batch_kernel/staged"}
    assert all(b["status"] == gbcg.CG_OK for b in out["batch"]), out["batch"]
