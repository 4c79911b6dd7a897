"""Column-sum pass at the ends of its chunks of samples (csrc/eval.cuh: 384 samples, 12
granules of 32): one, two, three and four chunks, full and with one sample in the last, so
that a buffer is used again; with few lanes per candidate (the order is checked every 32 or 64
samples) and with 8 and more (once per chunk). Tolerances as in test_gpu_parity."""
import numpy as np
import pytest

import workloads as W
from oracle import dls, models, varpro

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KS = [383, 384, 385, 767, 768, 769, 1151, 1152, 1153]
NS = [1, 2, 3, 6, 7, 8, 12, 13, 20]


@pytest.mark.parametrize("cb,lanes", [(64, 1), (32, 4), (16, 8), (4, 32)])
def test_column_sums_at_chunk_ends(cb, lanes):
    from paper_2109_01928_gb300 import debyefit as D
    P = 33   # a warp and more: fewer do not take a forced layout
    b = W.mixed_batch(S=len(KS), seed=19, P=P, K_range=(max(KS), max(KS)), N_range=(2, 12))
    keep = np.concatenate([np.arange(b.offsets[s], b.offsets[s] + k) for s, k in enumerate(KS)])
    re, im = models.synthesize(b)
    b.omega, re, im = b.omega[keep], re[keep], im[keep]
    b.offsets = np.concatenate([[0], np.cumsum(KS)]).astype(np.int64)
    b.n_poles[:] = NS
    th = W.population(b, P, seed=8)
    sp = D.make_spectra(b.offsets, b.omega, re, im, b.n_poles, b.lo, b.hi, device="cuda")
    theta = torch.as_tensor(th, device="cuda")
    with D.Handle("mixed", cands_per_block=cb, lanes_per_candidate=lanes) as h:
        cost = D.debye_eval_population(h, sp, theta).cpu().numpy()
        gcost, grad = D.debye_cost_grad(h, sp, theta)
        D.debye_sync(h)
    gcost, grad = gcost.cpu().numpy(), grad.cpu().numpy()
    for s in range(b.S):
        a, c = b.offsets[s], b.offsets[s + 1]
        om, N = b.omega[a:c], int(b.n_poles[s])
        ref, _ = dls.cost_population(om, re[a:c], im[a:c], th[s, :, :N])
        assert np.max(np.abs(cost[s] - ref) / ref) <= 1e-5, (s, KS[s], N)
        assert np.max(np.abs(gcost[s] - ref) / ref) <= 1e-5, (s, KS[s], N)
        for p in range(0, P, 16):
            x = dls.damped_solve(dls.basis(om, th[s, p, :N]), dls.target(re[a:c], im[a:c]), dls.LAM_SEARCH)
            if np.min(np.abs(x[1:])) < 1e-6 * np.abs(x).max():
                continue
            _, gref = varpro.cost_grad(om, re[a:c], im[a:c], th[s, p, :N])
            assert np.linalg.norm(grad[s, p, :N] - gref) <= 1e-4 * np.linalg.norm(gref), (s, p, KS[s], N)
