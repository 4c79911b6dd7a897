"""Input preparation of batches whose longest spectrum has more than 4096 samples: the planes
and granules are made by warps that find their spectrum by bisection, in turns of 4 places.
Spectra of 0, 1 and few samples beside long ones, in the first, middle and last place; costs
and gradients against the oracle (tolerances as in test_gpu_parity: 1e-5 and 1e-4), and bit
for bit against the same spectra in calls of their own, which a block per spectrum prepares
where they are short."""
import numpy as np
import pytest

import workloads as W
from oracle import dls, models, varpro

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BATCHES = [[4097], [1, 5000, 1], [33, 31, 32, 4100, 0, 0, 64, 127], [4099, 1, 1, 1, 1, 1, 1, 5], [2] * 40 + [9001],
           [4200, 4128, 4129, 50]]


@pytest.mark.parametrize("ks", BATCHES, ids=lambda k: "-".join(map(str, k[:4])))
def test_long_spectra_in_a_ragged_batch(ks):
    from paper_2109_01928_gb300 import debyefit as D
    S, P, top = len(ks), 32, max(ks)
    b = W.mixed_batch(S=S, seed=5, P=P, K_range=(top, top), N_range=(1, 4))
    # every spectrum thinned out to its own number of samples, over the whole band
    keep = [np.arange(k) * top // max(k, 1) for k in ks]
    idx = np.concatenate([b.offsets[s] + k for s, k in enumerate(keep)]).astype(np.int64)
    re, im = models.synthesize(b)
    om, re, im = b.omega[idx], re[idx], im[idx]
    offs = np.concatenate([[0], np.cumsum(ks)]).astype(np.int64)
    th = W.population(b, P, seed=4)
    theta = torch.as_tensor(th, device="cuda")
    with D.Handle("mixed", cands_per_block=32, lanes_per_candidate=1) as h:
        sp = D.make_spectra(offs, om, re, im, b.n_poles, b.lo, b.hi, device="cuda")
        D.debye_launch_count(h, reset=True)
        cost = D.debye_eval_population(h, sp, theta)
        groups = len(set(b.n_poles.tolist()))
        assert D.debye_launch_count(h) >= 2 + groups
        gcost, grad = D.debye_cost_grad(h, sp, theta)
        D.debye_sync(h)
        for s in range(S):
            a, c, N = offs[s], offs[s + 1], int(b.n_poles[s])
            if c == a:
                continue
            own = D.make_spectra([0, c - a], om[a:c], re[a:c], im[a:c], [N], [b.lo[s]], [b.hi[s]], device="cuda")
            one = theta[s:s + 1, :, :N].contiguous()
            assert torch.equal(D.debye_eval_population(h, own, one)[0], cost[s]), (s, ks[s])
            oc, og = D.debye_cost_grad(h, own, one)
            assert torch.equal(oc[0], gcost[s]) and torch.equal(og[0], grad[s, :, :N]), (s, ks[s])
            ref, _ = dls.cost_population(om[a:c], re[a:c], im[a:c], th[s, :, :N])
            assert np.max(np.abs(cost[s].cpu().numpy() - ref) / ref) <= 1e-5, (s, ks[s])
            if ks[s] <= 2:     # fewer rows than unknowns: the weights sit on flip kinks
                continue
            for p in (0, 17):
                x = dls.damped_solve(dls.basis(om[a:c], th[s, p, :N]), dls.target(re[a:c], im[a:c]), dls.LAM_SEARCH)
                if np.min(np.abs(x[1:])) < 1e-6 * np.abs(x).max():
                    continue
                _, gref = varpro.cost_grad(om[a:c], re[a:c], im[a:c], th[s, p, :N])
                assert np.linalg.norm(grad[s, p, :N].cpu().numpy() - gref) <= 1e-4 * np.linalg.norm(gref), (s, p)
        D.debye_sync(h)
