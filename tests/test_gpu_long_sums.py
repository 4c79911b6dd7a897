"""Column sums of very long spectra (csrc/eval.cuh, sums_write). The same-sign sums carry a bias
of 1 per lane, removed from the lanes' total in FP32: exact for any total that the pass can
reach, as an FP32 emulation shows on the CPU, and the cost of a spectrum of more than 2^24
samples, where one sample too many or too few moves it by several times the mixed precision's
tolerance, on the GPU."""
import numpy as np
import pytest


@pytest.mark.parametrize("ks", [1, 2, 4, 8, 16, 32])
def test_bias_removal_is_exact(ks):
    # one lane: sums of terms up to 1 stay at most 2^24; the total of ks lanes, as group_sum_ff
    # forms it; total - ks in FP32 against FP64
    f = np.float32
    rng = np.random.default_rng(ks)
    top = f(2 ** 24)
    for r in (f(1.0), np.nextafter(f(1.0), f(0.0)), f(0.75), f(0.5)):
        assert f(top + r) == top and f(np.nextafter(top, f(0.0)) + r) <= top
    n = 200000
    for lo, hi in ((1.0, 3.0), (1.0, 2.0 ** 24), (2.0 ** 22, 2.0 ** 24), (2.0 ** 24 - 64, 2.0 ** 24)):
        h = np.minimum(rng.uniform(lo, hi, (n, ks)).astype(f), top)
        h[: n // 10] = f(hi)
        while h.shape[1] > 1:
            h = (h[:, 0::2] + h[:, 1::2]).astype(f)
        t = h[:, 0]
        assert np.array_equal((t - f(ks)).astype(np.float64), t.astype(np.float64) - ks)


@pytest.mark.gpu
@pytest.mark.parametrize("K,cb,lanes", [((1 << 24) - 1, 32, 1), ((1 << 24) + 7, 32, 1), (30_000_000, 32, 1),
                                        ((1 << 24) + 7, 32, 2), ((1 << 25) + 3, 32, 4)])
def test_cost_of_a_long_spectrum(K, cb, lanes):
    # omega tau = 1e-13: the pole's column is the constant column, and against eps' = 1, eps'' = 0
    # the damped weights are 1 / (2 + lam) each, the cost K lam / (2 + lam). S off by one moves
    # it by 0.75, 9e-5 of it at 2^24 samples and 4.5e-5 at 2^25. (32 candidates: fewer do not
    # take a forced layout.)
    torch = pytest.importorskip("torch")
    from paper_2109_01928_gb300 import debyefit as D
    one = torch.ones(K, dtype=torch.float64, device="cuda")
    zero = torch.zeros(K, dtype=torch.float64, device="cuda")
    host = np.array([0, K], dtype=np.int64)
    t = lambda a, dt: torch.tensor(a, dtype=dt, device="cuda")
    sp = D.Spectra(t(host, torch.int64), one, one, zero, t([1], torch.int32), t([-13.5], torch.float64),
                   t([-12.5], torch.float64), host, np.array([1], dtype=np.int32))
    theta = torch.full((1, 32, 1), -13.0, dtype=torch.float64, device="cuda")
    with D.Handle("mixed", cands_per_block=cb, lanes_per_candidate=lanes) as h:
        lam = h.options.lam_search
        c, w = D.debye_eval_population(h, sp, theta, weights=True)
        g, _ = D.debye_cost_grad(h, sp, theta)
        D.debye_sync(h)
    ref = K * lam / (2 + lam)
    assert (c - ref).abs().max().item() <= 1e-5 * ref and (g - ref).abs().max().item() <= 1e-5 * ref
    assert torch.allclose(w.cpu(), torch.full((1, 32, 2), 1 / (2 + lam), dtype=torch.float64), rtol=1e-5, atol=0)
