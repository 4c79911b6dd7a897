"""The upload of a call's plan through the handle's pinned slots (csrc/host.h: four slots of
256 KB): more uploads in flight than slots, a plan larger than a slot, and a call refused
while the caller's stream is being captured. Work units decide which candidates a block takes
and in what order, not how a candidate is summed, so repeated calls give the same bits."""
import numpy as np
import pytest

import workloads as W
from oracle import dls, models

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _batch(D, S, K, N, P, seed):
    b = W.mixed_batch(S=S, seed=seed, P=P, K_range=K, N_range=N)
    re, im = models.synthesize(b)
    sp = D.make_spectra(b.offsets, b.omega, re, im, b.n_poles, b.lo, b.hi, device="cuda")
    th = W.population(b, P, seed=seed + 1)
    return b, re, im, sp, th, torch.as_tensor(th, device="cuda")


def _check(b, re, im, th, cost, spectra):
    for s in spectra:
        a, c = b.offsets[s], b.offsets[s + 1]
        ref, _ = dls.cost_population(b.omega[a:c], re[a:c], im[a:c], th[s, :, :int(b.n_poles[s])])
        assert np.max(np.abs(cost[s] - ref) / ref) <= 1e-5, s


@pytest.mark.parametrize("prec", ["mixed", "mixed_table", "fp64"])
def test_more_uploads_in_flight_than_slots(prec):
    # long evaluations keep the stream busy while a dozen calls of different plans queue up
    from paper_2109_01928_gb300 import debyefit as D
    long = _batch(D, 40, (2000, 2000), (8, 8), 512, 1)
    small = [_batch(D, 3 + 5 * i, (10, 60), (1, 1 + i), 9 + i, 10 * i) for i in range(12)]
    with D.Handle(prec) as h:
        alone = []
        for x in small:
            alone.append(D.debye_eval_population(h, x[3], x[5]))
            torch.cuda.synchronize()
        D.debye_eval_population(h, long[3], long[5])
        torch.cuda.synchronize()
        for _ in range(6):
            D.debye_eval_population(h, long[3], long[5])
        queued = [D.debye_eval_population(h, x[3], x[5]) for x in small]
        D.debye_sync(h)
    for x, a, q in zip(small, alone, queued):
        assert torch.equal(a, q)
        _check(x[0], x[1], x[2], x[4], q.cpu().numpy(), range(x[0].S))


def test_a_plan_larger_than_a_slot():
    # 9000 spectra, a work unit of 32 bytes each: 288 KB; small plans before and after
    from paper_2109_01928_gb300 import debyefit as D
    small = _batch(D, 5, (10, 60), (1, 4), 12, 3)
    large = _batch(D, 9000, (2, 4), (1, 3), 2, 5)
    with D.Handle("mixed") as h:
        first = D.debye_eval_population(h, small[3], small[5])
        costs = [D.debye_eval_population(h, large[3], large[5]) for _ in range(6)]   # every slot grows
        again = D.debye_eval_population(h, small[3], small[5])
        D.debye_sync(h)
    assert torch.equal(first, again)
    for c in costs[1:]:
        assert torch.equal(costs[0], c)
    _check(large[0], large[1], large[2], large[4], costs[0].cpu().numpy(), range(0, 9000, 997))


def test_refused_under_capture():
    # a replay would copy whatever the slot holds by then: the call fails, the capture and the
    # handle stay usable
    from paper_2109_01928_gb300 import debyefit as D
    b, re, im, sp, th, theta = _batch(D, 4, (20, 50), (2, 3), 16, 7)
    with D.Handle("mixed") as h:
        ref = D.debye_eval_population(h, sp, theta)
        torch.cuda.synchronize()
        out = torch.empty_like(ref)
        x = torch.zeros(8, device="cuda")
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            with pytest.raises(D.DebyeError) as e:
                D.debye_eval_population(h, sp, theta, cost=out)
            x += 1
        assert e.value.code == D.DEBYE_ECUDA
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(x, torch.ones_like(x))
        again = D.debye_eval_population(h, sp, theta)
        D.debye_sync(h)
    assert torch.equal(ref, again)
