"""The search kernels at the sizes where their paths change: populations around the block
(256) and the limit of the fused swarm step (1024), coefficients that are powers of two and
that are not; the polish's rounds (8 step lengths, or every one at once); table boxes read
from shared memory and from where they are."""
import numpy as np
import pytest

import workloads as W
from oracle import dls, models, pso

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [3, 255, 257, 1024, 1025, 1500])
@pytest.mark.parametrize("coef", [(0.5, 0.5, 0.5), (0.7298, 0.25, 1.49618)])
def test_swarm_trace_follows_oracle(P, coef):
    # FP64 costs agree to 1e-10 (their parity tolerance) and the update is bit-identical, so
    # the traces agree to 1e-10 over a few generations
    from paper_2109_01928_gb300 import debyefit as D
    b = W.mixed_batch(S=2, seed=17, P=P, K_range=(20, 40), N_range=(1, 3))
    re, im = models.synthesize(b)
    om, pp, pg = coef
    with D.Handle("fp64", pso_omega=om, pso_phi_p=pp, pso_phi_g=pg) as h:
        sp = D.make_spectra(b.offsets, b.omega, re, im, b.n_poles, b.lo, b.hi, device="cuda")
        out = D.debye_fit_batch(h, sp, P=P, iters=5, seed=3, polish_topk=0, trace=True)
        D.debye_sync(h)
    tr = out["trace"].cpu().numpy()
    for s in range(b.S):
        a, c = b.offsets[s], b.offsets[s + 1]
        cost = lambda th: dls.cost_population(b.omega[a:c], re[a:c], im[a:c], th)[0]
        _, _, _, ref = pso.pso(cost, int(b.n_poles[s]), b.lo[s], b.hi[s], P, 5, seed=3, spectrum=s, omega=om,
                               phi_p=pp, phi_g=pg)
        np.testing.assert_allclose(tr[s], ref, rtol=1e-10, atol=0)
    assert out["evals"].item() == P * 6 * b.omega.shape[0]


@pytest.mark.parametrize("prec", ["mixed", "mixed_table", "fp64"])
@pytest.mark.parametrize("trials", [1, 2, 9, 20, 33, 40])
def test_polish_rounds_give_one_result(prec, trials):
    # a failure counter keeps the rounds of 8 step lengths; without one a small batch takes
    # every step length in one round: the same line search, so the same bits
    from paper_2109_01928_gb300 import debyefit as D
    b = W.mixed_batch(S=5, seed=29, P=32, K_range=(30, 200), N_range=(2, 12))
    re, im = models.synthesize(b)
    res = []
    for n_failed in (True, False):
        with D.Handle(prec, lbfgs_max_trials=trials) as h:
            sp = D.make_spectra(b.offsets, b.omega, re, im, b.n_poles, b.lo, b.hi, device="cuda")
            out = D.debye_fit_batch(h, sp, P=32, iters=3, seed=1, polish_topk=5, polish_iters=12, n_failed=n_failed)
            D.debye_sync(h)
        res.append({k: out[k].cpu().numpy() for k in ("eps_inf", "d_eps", "tau", "final_cost", "evals")})
    for k in res[0]:
        assert np.array_equal(res[0][k], res[1][k]), k


@pytest.mark.parametrize("span", [0.15, 8.0, 12.8, 13.0, 21.0])
def test_table_boxes_staged_and_not(span):
    # 1, 40 and 64 segments are copied to shared memory for 64 candidates, 65 and 105 are
    # read in place, as any are for 3 candidates (fewer than two poles per segment): the
    # same polynomials, so the same bits
    from paper_2109_01928_gb300 import debyefit as D
    b = W.mixed_batch(S=3, seed=31, P=64, K_range=(40, 90), N_range=(2, 6))
    b.lo[:] = -14.0
    b.hi[:] = -14.0 + span
    re, im = models.synthesize(b)
    sp = D.make_spectra(b.offsets, b.omega, re, im, b.n_poles, b.lo, b.hi, device="cuda")
    theta = torch.as_tensor(W.population(b, 64, seed=6), device="cuda")
    with D.Handle("mixed_table") as h:
        many = D.debye_eval_population(h, sp, theta, weights=True)
        few = D.debye_eval_population(h, sp, theta[:, :3].contiguous(), weights=True)
        D.debye_sync(h)
    assert torch.equal(many[0][:, :3], few[0]) and torch.equal(many[1][:, :3], few[1])
    assert torch.isfinite(many[0]).all()
