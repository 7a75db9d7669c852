"""Mini-batches spread over the training lanes (streams) against the pairs one
by one: batches smaller than, equal to and larger than the lanes, pairs of
several instances, repeated pairs."""
import numpy as np
import pytest

from paper_1107_0538_gb300 import gbcg, problems

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("e", [5, 17])
def test_batch_gradient_is_the_mean_of_its_pairs(e):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    inst = [problems.learn_instance(e, 30000 + i) for i in range(3)]
    net = gbcg.Net(problems.learn_init_params())
    solvers, R, E, pi = [], [], [], []
    for k, it in enumerate(inst):
        s = gbcg.Solver(it.A, precond=gbcg.CG_PRECOND_LEARNED)
        s.set_learned(net, it.grid, it.lognu.astype(np.float32))
        r = torch.empty((2, it.A.n), dtype=torch.float32, device=dev)
        er = torch.empty_like(r)
        s.learn_pairs(torch.from_numpy(it.b).to(dev), torch.from_numpy(it.xstar).to(dev), 4, 2, r, er)
        solvers.append(s)
        R.append(r)
        E.append(er)
        pi += [k, k]
    lset = gbcg.LearnSet(solvers, np.array(pi, np.int32), torch.cat(R).contiguous(), torch.cat(E).contiguous())
    one = [net.grad(lset, [k]) for k in range(6)]
    for pairs in ([0], [0, 3], [5, 1, 2, 0], [0, 1, 2, 3, 4], [4, 4, 1, 0, 5, 2, 3, 3, 1]):
        loss, g = net.grad(lset, pairs)
        want_l = np.mean([one[k][0] for k in pairs])
        want_g = np.mean([one[k][1].astype(np.float64) for k in pairs], axis=0)
        # the pairs' own gradients carry FP32 sums of up to a few thousand terms
        # in another order: 2^-24 times the root of that, doubled twice
        assert abs(loss - want_l) <= 1e-12 * abs(want_l)
        assert np.linalg.norm(g - want_g) <= 4 * 2.0 ** -24 * 64 * np.linalg.norm(want_g)
        again = net.grad(lset, pairs)
        assert again[0] == loss and np.array_equal(again[1], g)
    for s in solvers:
        s.close()
    net.close()
