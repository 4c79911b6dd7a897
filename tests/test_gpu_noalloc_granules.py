"""The allocation-free entry point where the granule records do not fit after the sample planes
(csrc/noalloc.cu: hardly more samples than spectra) and take the factor's memory: spectra of
one sample, one candidate of one pole each, where the margin is smallest (24 bytes against
16.5 per spectrum). Either entry point is within its precision's tolerance of the oracle, so
they are within twice that of each other."""
import numpy as np
import pytest

import workloads as W
from oracle import dls, models

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("S,P,longer", [(1, 1, 0), (31, 1, 0), (32, 1, 0), (33, 1, 1), (33, 1, 2), (1000, 1, 0),
                                        (1000, 1, 31), (1000, 1, 32), (70, 3, 2), (4096, 1, 0)])
def test_one_sample_per_spectrum(prec, S, P, longer):
    # `longer` spectra have two samples: with n samples, n / 32 + S records, the fallback ends
    # where n >= S + n / 32
    from paper_2109_01928_gb300 import debyefit as D
    K = np.ones(S, dtype=np.int64)
    K[:longer] = 2
    b = W.mixed_batch(S=S, seed=23, P=P, K_range=(2, 2), N_range=(1, 1))
    re, im = models.synthesize(b)
    keep = np.concatenate([np.arange(b.offsets[s], b.offsets[s] + k) for s, k in enumerate(K)])
    om, re, im = b.omega[keep], re[keep], im[keep]
    offs = np.concatenate([[0], np.cumsum(K)]).astype(np.int64)
    sp = D.make_spectra(offs, om, re, im, b.n_poles, b.lo, b.hi, device="cuda")
    th = W.population(b, P, seed=2)
    theta = torch.as_tensor(th, device="cuda")
    tol = 1e-10 if prec == "fp64" else 1e-5
    with D.Handle(prec) as h:
        ref = D.debye_eval_population(h, sp, theta).cpu().numpy()
        D.debye_sync(h)
    for _ in range(2):
        c = D.debye_eval_population_noalloc(sp, theta, precision=prec).cpu().numpy()
        assert np.max(np.abs(c - ref) / ref) <= 2 * tol
        for s in range(0, S, max(1, S // 40)):
            a, e = offs[s], offs[s + 1]
            o, _ = dls.cost_population(om[a:e], re[a:e], im[a:e], th[s, :, :1])
            assert np.max(np.abs(c[s] - o) / o) <= tol, s
