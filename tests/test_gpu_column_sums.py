"""Column-sum pass at the sizes where its paths change: granules and chunks of samples
(32 and 128) and their remainders, odd and even pole counts below, at and above one
sweep, several lanes per candidate; and the sample orders and signs that decide between
its ordered and its general exact sums (ascending, descending and shuffled frequencies,
eps'' of either sign). Tolerances as in test_gpu_parity: 1e-5 on mixed costs, 1e-4 on
gradients (norm-wise per candidate, away from flip kinks)."""
import numpy as np
import pytest

import workloads as W
from oracle import dls, models, varpro

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KS = [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 257, 400]
NS = [1, 2, 3, 6, 7, 8, 9, 12, 13, 16, 17, 19, 20, 5]


def _reorder(b, re, im, order, rng):
    om = b.omega.copy()
    re, im = re.copy(), im.copy()
    for s in range(b.S):
        a, c = b.offsets[s], b.offsets[s + 1]
        K = c - a
        idx = np.arange(K)[::-1] if order == "descending" else rng.permutation(K) if order == "shuffled" else np.arange(K)
        om[a:c], re[a:c], im[a:c] = om[a:c][idx], re[a:c][idx], im[a:c][idx]
        if order == "signs":        # the second half of the spectra: eps'' (and some eps') of either sign
            if s % 2:
                im[a:c] *= rng.choice([-1.0, 1.0], K)
                re[a:c] *= np.where(rng.random(K) < 0.1, -1.0, 1.0)
    return om, re, im


@pytest.mark.parametrize("order", ["ascending", "descending", "shuffled", "signs"])
@pytest.mark.parametrize("cb,lanes", [(0, 0), (64, 1), (32, 4)])
def test_column_sums_edges(order, cb, lanes):
    from paper_2109_01928_gb300 import debyefit as D
    rng = np.random.default_rng(5)
    P = 34
    b = W.mixed_batch(S=len(KS), seed=9, P=P, K_range=(400, 400), N_range=(2, 12))
    keep = np.concatenate([np.arange(b.offsets[s], b.offsets[s] + k) for s, k in enumerate(KS)])
    re, im = models.synthesize(b)
    b.omega, re, im = b.omega[keep], re[keep], im[keep]
    b.offsets = np.concatenate([[0], np.cumsum(KS)]).astype(np.int64)
    b.n_poles[:] = NS
    om, re, im = _reorder(b, re, im, order, rng)
    th = W.population(b, P, seed=4)
    sp = D.make_spectra(b.offsets, om, re, im, b.n_poles, b.lo, b.hi, device="cuda")
    theta = torch.as_tensor(th, device="cuda")
    with D.Handle("mixed", cands_per_block=cb, lanes_per_candidate=lanes) as h:
        cost = D.debye_eval_population(h, sp, theta).cpu().numpy()
        gcost, grad = D.debye_cost_grad(h, sp, theta)
        D.debye_sync(h)
    gcost, grad = gcost.cpu().numpy(), grad.cpu().numpy()
    for s in range(b.S):
        a, c = b.offsets[s], b.offsets[s + 1]
        N = int(b.n_poles[s])
        ref, _ = dls.cost_population(om[a:c], re[a:c], im[a:c], th[s, :, :N])
        assert np.max(np.abs(cost[s] - ref) / ref) <= 1e-5, (s, KS[s], N)
        assert np.max(np.abs(gcost[s] - ref) / ref) <= 1e-5, (s, KS[s], N)
        if KS[s] <= 2:          # fewer rows than unknowns: the weights sit on flip kinks
            continue
        for p in range(0, P, 11):
            x = dls.damped_solve(dls.basis(om[a:c], th[s, p, :N]), dls.target(re[a:c], im[a:c]), dls.LAM_SEARCH)
            if np.min(np.abs(x[1:])) < 1e-6 * np.abs(x).max():
                continue
            _, gref = varpro.cost_grad(om[a:c], re[a:c], im[a:c], th[s, p, :N])
            assert np.linalg.norm(grad[s, p, :N] - gref) <= 1e-4 * np.linalg.norm(gref), (s, p, KS[s], N)
