"""Column-sum tables at the node counts where the node pass's blocks change: boxes of one
segment (12 nodes, two groups of 6) up to several full blocks of 16 groups and their
remainders (8 segments fill one block, 9 start a second), few samples and many. Costs and
gradients against the oracle, tolerances as in test_gpu_parity: 1e-5 on costs, 1e-4 on
gradients (norm-wise per candidate, away from flip kinks)."""
import numpy as np
import pytest

import workloads as W
from oracle import dls, models, varpro

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SEGS = [1, 2, 7, 8, 9, 15, 16, 17, 24, 40, 41]


@pytest.mark.parametrize("K", [5, 129, 700])
def test_table_node_blocks(K):
    from paper_2109_01928_gb300 import debyefit as D
    S, P = len(SEGS), 20
    b = W.mixed_batch(S=S, seed=31, P=P, K_range=(K, K), N_range=(2, 4))
    b.lo[:] = -12.5
    b.hi[:] = b.lo + 0.2 * np.array(SEGS) - 0.05
    re, im = models.synthesize(b)
    th = W.population(b, P, seed=6)
    sp = D.make_spectra(b.offsets, b.omega, re, im, b.n_poles, b.lo, b.hi, device="cuda")
    theta = torch.as_tensor(th, device="cuda")
    with D.Handle("mixed_table") as h:
        cost = D.debye_eval_population(h, sp, theta).cpu().numpy()
        gcost, grad = D.debye_cost_grad(h, sp, theta)
        D.debye_sync(h)
    gcost, grad = gcost.cpu().numpy(), grad.cpu().numpy()
    for s in range(S):
        a, c = b.offsets[s], b.offsets[s + 1]
        N = int(b.n_poles[s])
        om, er, ei = b.omega[a:c], re[a:c], im[a:c]
        ref, _ = dls.cost_population(om, er, ei, th[s, :, :N])
        assert np.max(np.abs(cost[s] - ref) / ref) <= 1e-5, (s, SEGS[s], N)
        assert np.max(np.abs(gcost[s] - ref) / ref) <= 1e-5, (s, SEGS[s], N)
        for p in range(0, P, 7):
            x = dls.damped_solve(dls.basis(om, th[s, p, :N]), dls.target(er, ei), dls.LAM_SEARCH)
            if np.min(np.abs(x[1:])) < 1e-6 * np.abs(x).max():
                continue
            _, gref = varpro.cost_grad(om, er, ei, th[s, p, :N])
            assert np.linalg.norm(grad[s, p, :N] - gref) <= 1e-4 * np.linalg.norm(gref), (s, p, SEGS[s], N)
