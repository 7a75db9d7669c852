"""The learned preconditioner's application where its tensor-core convolution
gives a CTA several bricks of 8 x 16 x 4 outputs (two staging buffers and two
accumulator sets take turns), against the FP64 oracle, brick by brick.

The network runs in BF16 with FP32 accumulation: six roundings in sequence of
at most 2^-9 each, 1.2e-2 of the normwise result.  Within one brick the terms of
a sum may cancel up to tenfold against the norm of the whole, so a brick's
error must stay below 10 * 1.2e-2 of the larger of its own norm and the field's
mean brick norm; a brick computed from the wrong data is off by about 1."""
import numpy as np
import pytest

from oracle import learn as OL
from paper_1107_0538_gb300 import gbcg, problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# elements per axis: fewer bricks than CTAs (304 on 152 SMs), some CTAs with two,
# an odd and an even number of rounds, ragged ends of one node in every axis
DIMS = [(16, 16, 4), (79, 79, 27), (80, 64, 28), (64, 80, 64), (87, 79, 47)]


@pytest.mark.parametrize("dims", DIMS, ids=lambda d: "x".join(map(str, d)))
def test_apply_matches_oracle_in_every_brick(dims):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ex, ey, ez = dims
    grid = P.Grid(ex, ey, ez, 1.0 / max(dims))
    nu = P.nu_blobs(grid, seed=31, nu_iron=1e-3)
    A, _ = P.q1_matrix(nu, grid.h)
    lognu = P.node_log_nu(grid, nu).astype(np.float32)
    rng = np.random.default_rng(17)
    th = P.learn_init_params(seed=5, noise=0.3).astype(np.float64)
    th[OL.N_W1 + OL.N_W2:OL.N_W1 + OL.N_W2 + OL.N_WG] = 0.5 * rng.standard_normal(OL.N_WG)
    th = P.bf16_representable(th)
    r = rng.standard_normal(A.n)
    shape = (ez + 1, ey + 1, ex + 1)
    ref = OL.apply(th, r, OL.diagonal(A), lognu.astype(np.float64), shape).reshape(shape)
    with gbcg.Solver(A, precond=gbcg.CG_PRECOND_LEARNED) as s:
        s.set_learned(gbcg.Net(th.astype(np.float32)), grid, lognu)
        rt = torch.from_numpy(r).to("cuda:0")
        zt = torch.zeros_like(rt)
        s.precond_apply(rt, zt)
        z = zt.cpu().numpy().reshape(shape)
    assert np.linalg.norm(z - ref) <= 3e-2 * np.linalg.norm(ref)
    cut = [range(0, n, b) for n, b in zip(shape, (4, 16, 8))]
    bricks = [(slice(k, k + 4), slice(j, j + 16), slice(i, i + 8)) for k in cut[0] for j in cut[1] for i in cut[2]]
    rms = np.sqrt(np.mean(ref * ref))
    for b in bricks:
        scale = max(np.linalg.norm(ref[b]), rms * np.sqrt(ref[b].size))
        assert np.linalg.norm(z[b] - ref[b]) <= 0.12 * scale, b
