"""The work a user of the library has it do, as timed cases.

A case is one call of a public entry point on one batch of spectra: an evaluation of a
population of candidates (costs, optionally the weights), an evaluation with the
gradient, or a whole fit. Targets are computed here, in plain torch (FP64), from the
relaxation models and parameter ranges of the named workloads; populations are half
uniform in the search box (a first generation) and half gathered around one point per
spectrum (a swarm that has begun to converge).
"""
import math

import numpy as np
import torch

from paper_2109_01928_gb300 import debyefit as D

LAM = 1e-3          # the library's default damping
LN10 = math.log(10.0)


def _case(name, kind, batch, S, K, N, P, precision, **more):
    """K and N are ranges [lo, hi], drawn per spectrum."""
    c = {"kind": kind, "batch": batch, "S": S, "K_lo": K[0], "K_hi": K[1], "N_lo": N[0], "N_hi": N[1], "P": P,
         "precision": precision}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # One measured spectrum, one small population: the smallest call a program makes
        # (a hand-written search around the library). All launches and host work.
        _case("eval_single_k50", "eval", "hn", 1, (50, 50), (3, 3), 64, "mixed"),
        # A ragged batch with odd sizes, from two samples and one pole up to the largest
        # pole count, with the weights: the general call with no size that fits a tile.
        _case("eval_ragged_odd", "eval", "mixed", 61, (2, 701), (1, 20), 37, "mixed", weights=True),
        # One generation of the 1024-spectrum workload: what a search does over and over.
        _case("eval_mixed_1024", "eval", "mixed", 1024, (50, 1000), (2, 12), 256, "mixed"),
        # Densely sampled tabulated spectra with the most poles: the longest sums.
        _case("eval_tabulated_k4096", "eval", "tabulated", 512, (4096, 4096), (20, 20), 512, "mixed"),
        # The same generation in the table precision.
        _case("eval_table_1024", "eval", "mixed", 1024, (50, 1000), (2, 12), 256, "mixed_table"),
        # FP64 with column sums, with the weights.
        _case("eval_fp64_sums_256", "eval", "mixed", 256, (50, 1000), (2, 12), 256, "fp64_sums", weights=True),
        # Differentiation of a large fed-in population (gradient-based search): the largest work.
        _case("grad_hn_k2000", "grad", "hn", 256, (2000, 2000), (8, 8), 4096, "mixed"),
        # Few candidates per spectrum with their gradients: the points of a local search.
        _case("grad_points_1024", "grad", "mixed", 1024, (50, 1000), (2, 12), 8, "mixed"),
        # The plain FP64 method with its gradient.
        _case("grad_fp64_256", "grad", "mixed", 256, (50, 1000), (2, 12), 64, "fp64"),
        # The paper's use: fit one spectrum (seeded swarm, then the local polish).
        _case("fit_single_k50", "fit", "hn", 1, (50, 50), (3, 3), 64, "mixed", method="pso", iters=100, topk=8,
              polish=50),
        # The whole fit of the 1024-spectrum workload, in the default precision ...
        _case("fit_mixed_1024", "fit", "mixed", 1024, (50, 1000), (2, 12), 256, "mixed", method="pso", iters=200,
              topk=8, polish=50),
        # ... and in the table precision.
        _case("fit_table_1024", "fit", "mixed", 1024, (50, 1000), (2, 12), 256, "mixed_table", method="pso",
              iters=200, topk=8, polish=50),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, batch and precision, sizes log-uniform over their ranges,
    cut so that it costs no more than the listed ones."""
    kind = rng.choice(["eval", "eval", "eval", "grad", "grad", "fit"])
    batch = rng.choice(["mixed", "mixed", "hn", "tabulated"])
    precision = rng.choice(["mixed", "mixed", "mixed", "mixed_table", "mixed_table", "fp64", "fp64_sums"])
    S, P = _log(rng, 1, 1024), _log(rng, 4 if kind == "grad" else 16, 4096 if kind != "fit" else 256)
    if batch == "mixed":
        k0 = _log(rng, 2, 400)
        K = (k0, max(k0, _log(rng, 50, 1000)))
        n0 = rng.randint(1, 12)
        N = (n0, rng.randint(n0, 20))
    else:
        k0 = _log(rng, 20, 4096 if batch == "tabulated" else 2000)
        n0 = rng.randint(1, 20)
        K, N = (k0, k0), (n0, n0)
    more = {}
    # poles x samples x candidates of one pass, at most a part of the largest listed cases'
    cap = {"mixed": 4e9, "mixed_table": 4e9, "fp64": 4e7, "fp64_sums": 1.5e8}[precision]
    evals = 1
    if kind == "eval":
        more["weights"] = bool(rng.randint(0, 1))
    if kind == "fit":
        more = {"method": rng.choice(["pso", "pso", "de", "da"]), "iters": rng.randint(10, 100),
                "topk": rng.choice([0, 1, 4, 8]), "polish": rng.randint(5, 50)}
        if more["method"] == "da":
            more["iters"] = rng.randint(3, 10)
        evals = more["iters"] * (2 * N[1] if more["method"] == "da" else 1) + 8 * more["polish"]
        cap *= 8
    mean = 0.25 * (K[0] + K[1]) * (N[0] + N[1])
    while S > 1 and S * P * mean * evals > cap:
        S = max(1, S * 3 // 4)
    while P > 8 and S * P * mean * evals > cap:
        P = max(8, P * 3 // 4)
    return _case(None, kind, batch, S, K, N, P, precision, **more)


# ------------------------------------------------------------------ inputs

def _shape(case):
    """Sample and pole counts of every spectrum: part of the case, not of the seed."""
    r = np.random.default_rng([case["S"], case["K_lo"], case["K_hi"], case["N_lo"], case["N_hi"]])
    S = case["S"]
    K = r.integers(case["K_lo"], case["K_hi"] + 1, S)
    N = r.integers(case["N_lo"], case["N_hi"] + 1, S)
    if case["K_hi"] > case["K_lo"] and S > 1:
        K[0], N[0] = case["K_lo"], case["N_hi"]
    return K, N


def _inputs(case, seed):
    """Host arrays of the batch (offsets, omega, eps', eps'', n_poles, lo, hi) and, for the
    evaluations, the population on the GPU."""
    r = np.random.default_rng([seed, 11])
    S = case["S"]
    K, N = _shape(case)
    offs = np.concatenate([[0], np.cumsum(K)]).astype(np.int64)
    dev = "cuda"
    t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=dev)
    sid = torch.as_tensor(np.repeat(np.arange(S), K), device=dev)
    pos = torch.arange(int(offs[-1]), device=dev) - torch.as_tensor(offs[:-1], device=dev)[sid]
    f0, f1 = (1e8, 1e10) if S == 1 and case["batch"] == "hn" else (1e5 if case["batch"] == "tabulated" else 1e6, 1e10)
    frac = pos.double() / torch.clamp(t(K - 1.0)[sid], min=1.0)
    om = 2 * math.pi * 10.0 ** (math.log10(f0) + (math.log10(f1) - math.log10(f0)) * frac)
    eps_inf = t(r.uniform(2.0, 8.0, S))[sid]
    jw = torch.complex(torch.zeros_like(om), om)

    def power(z, p):
        return torch.polar(z.abs() ** p, z.angle() * p)

    def hn(d, tau, al, be):
        one = torch.ones((), dtype=torch.complex128, device=dev)
        return eps_inf + t(d)[sid] / power(one + power(jw * t(tau)[sid], t(al)[sid]), t(be)[sid])

    def jonscher(a, n):
        g = t(a)[sid] * (om / (2 * math.pi * 1e8)) ** (t(n)[sid] - 1.0)
        return torch.complex(g, -g / torch.tan(t(n)[sid] * (math.pi / 2)))

    d = r.uniform(1.0, 80.0, S)
    tau = 10.0 ** r.uniform(-11.0, -8.0, S)
    al, be = r.uniform(0.3, 1.0, S), r.uniform(0.3, 1.0, S)
    a_p, n_p = r.uniform(1.0, 10.0, S), r.uniform(0.3, 0.9, S)
    if case["batch"] == "tabulated":
        # "measured" spectra: 40 Debye poles, a Jonscher tail and 1 % noise
        eps = eps_inf + jonscher(a_p, n_p)
        pt, pd = 10.0 ** r.uniform(-12.0, -6.0, (S, 40)), 10.0 ** r.uniform(-1.0, math.log10(20.0), (S, 40))
        for j in range(40):
            eps = eps + t(pd[:, j])[sid] / (1.0 + jw * t(pt[:, j])[sid])
        g = torch.Generator(device=dev).manual_seed(seed)
        z = torch.randn(2, om.numel(), dtype=torch.float64, device=dev, generator=g)
        er, ei = eps.real * (1 + 0.01 * z[0]), -eps.imag * (1 + 0.01 * z[1])
    else:
        if case["batch"] == "mixed":   # Havriliak-Negami, Cole-Cole, Cole-Davidson, Jonscher, CRIM
            model = r.integers(0, 5, S)
            be = np.where(model == 1, 1.0, be)
            al = np.where(model == 2, 1.0, al)
            fr = r.dirichlet([1.0, 1.0, 1.0], S)
            water = 4.9 + 75.0 / (1.0 + jw * 9.23e-12)
            crim = power(t(fr[:, 0])[sid] * power(water, torch.full_like(om, 0.5)) + t(fr[:, 1])[sid] * math.sqrt(4.5)
                         + t(fr[:, 2])[sid], torch.full_like(om, 2.0))
            m = torch.as_tensor(model, device=dev)[sid]
            eps = torch.where(m < 3, hn(d, tau, al, be),
                              torch.where(m == 3, eps_inf + jonscher(a_p, n_p), crim))
        else:
            eps = hn(d, tau, al, be)
        er, ei = eps.real, -eps.imag
    lo, hi = np.full(S, -13.0), np.full(S, -6.0 if S == 1 and case["batch"] == "hn" else -5.0)
    host = (offs, om.cpu().numpy(), er.cpu().numpy(), ei.cpu().numpy(), N.astype(np.int32), lo, hi)
    theta = None
    if case["kind"] != "fit":
        P, nmax = case["P"], int(N.max())
        g = torch.Generator(device=dev).manual_seed(seed + 1)
        u = torch.rand(S, P, nmax, dtype=torch.float64, device=dev, generator=g)
        lo_t, hi_t = t(lo)[:, None, None], t(hi)[:, None, None]
        theta = lo_t + (hi_t - lo_t) * u
        near = theta[:, :1] + 0.3 * torch.randn(S, P, nmax, dtype=torch.float64, device=dev, generator=g)
        half = (torch.arange(P, device=dev) >= P // 2)[None, :, None]
        theta = torch.minimum(torch.maximum(torch.where(half, near, theta), lo_t), hi_t)
        keep = torch.arange(nmax, device=dev)[None, None, :] < torch.as_tensor(N, device=dev)[:, None, None]
        theta = torch.where(keep, theta, torch.zeros_like(theta)).contiguous()
    return host, theta


def prepare(case, seed):
    """The spectra on the GPU, a handle, and the population (or, for a fit, the seed)."""
    host, theta = _inputs(case, seed)
    return {"case": case, "h": D.Handle(case["precision"]), "sp": D.make_spectra(*host), "theta": theta, "seed": seed}


def run(state):
    c, h, sp = state["case"], state["h"], state["sp"]
    if c["kind"] == "eval":
        return D.debye_eval_population(h, sp, state["theta"], weights=c.get("weights", False))
    if c["kind"] == "grad":
        return D.debye_cost_grad(h, sp, state["theta"])
    return D.debye_fit_batch(h, sp, P=c["P"], iters=c["iters"], seed=state["seed"], polish_topk=c["topk"],
                             polish_iters=c["polish"], method=c["method"])


def work(case):
    """Bytes: spectra and thetas in, results out. FLOPs: per candidate, sample and pole the
    basis value and the sums it enters (1 / (1 + w^2 tau^2), its sum and two products; the
    same sums again for the derivative columns with a gradient), per candidate the damped
    solve of N + 1 unknowns. The table precision's sums do not grow with the samples per
    candidate: its samples enter only the table (12 nodes on each of 40 segments, with the
    derivative sums)."""
    K, N = (a.astype(np.float64) for a in _shape(case))
    S, P, nmax = case["S"], case["P"], int(N.max())
    grad = case["kind"] == "grad"
    table = case["precision"] == "mixed_table"
    per = 16.0 if grad else 8.0
    one = float(np.sum(P * K * N)) * (0.0 if table else per)     # one evaluation's sums
    if table:
        one = float(np.sum(P * N)) * 24.0 * 3.0
    one += float(np.sum(P * ((N + 1) ** 3 / 3.0 + 4.0 * (N + 1) ** 2))) * (2.0 if grad else 1.0)
    build = float(np.sum(K)) * 480.0 * 16.0 if table else 0.0
    nbytes = 24.0 * float(K.sum())
    if case["kind"] == "fit":
        moves = case["iters"] * (2.0 * float(N.mean()) if case["method"] == "da" else 1.0) + 1.0
        polish = min(case["topk"], P) / P * (case["polish"] + 1.0) * 2.0
        return {"bytes": nbytes + 8.0 * S * (2 * nmax + 2), "flops": build + one * (moves + polish)}
    nbytes += 8.0 * S * P * (nmax + 1)
    if grad:
        nbytes += 8.0 * S * P * nmax
    if case.get("weights"):
        nbytes += 8.0 * S * P * (nmax + 1)
    return {"bytes": nbytes, "flops": build + one}


# ------------------------------------------------------------------ 64-bit values

def _cost64(om, er, ei, theta, want):
    """Damped cost, flipped weights and (want == "grad") the gradient of theta [P, N], by the
    plain method: basis, normal equations, solve, flip, misfit; the gradient by autograd."""
    th = theta.clone().requires_grad_(want == "grad")
    x = om[None, :, None] * 10.0 ** th[:, None, :]
    re = 1.0 / (1.0 + x * x)
    im = x * re
    P, K, N = re.shape
    ones, zeros = re.new_ones(P, K, 1), re.new_zeros(P, K, 1)
    A = torch.cat([torch.cat([ones, re], 2), torch.cat([zeros, im], 2)], 1)
    b = torch.cat([er, ei])
    G = A.transpose(1, 2) @ A
    g = torch.diagonal(G, dim1=1, dim2=2)
    s = torch.rsqrt(g)
    C = G * s[:, :, None] * s[:, None, :] + LAM * torch.eye(N + 1, dtype=torch.float64, device=om.device)
    y = torch.linalg.solve(C, (s * (A.transpose(1, 2) @ b))[..., None])[..., 0] * s
    flip = torch.cat([torch.ones_like(y[:, :1]), torch.where(y[:, 1:] < 0, -1.0, 1.0).to(y)], 1)
    xh = y * flip.detach()
    r = (A @ xh[..., None])[..., 0] - b
    cost = (r * r).sum(1) + LAM * (g * xh * xh).sum(1)
    grad = torch.autograd.grad(cost.sum(), th)[0] if want == "grad" else None
    return cost.detach(), xh.detach(), grad


def exact(case, seed):
    """The outputs of run() in 64 bits; None for the whole fits (a search and a local polish,
    whose path is not a computed number)."""
    if case["kind"] == "fit":
        return None
    K, N = _shape(case)
    if float(np.sum(case["P"] * K * N * (N + 1.0))) > 3e11:   # beyond about 20 s
        return None
    (offs, om, er, ei, _, _, _), theta = _inputs(case, seed)
    om, er, ei = (torch.as_tensor(a, device="cuda") for a in (om, er, ei))
    S, P, nmax = theta.shape
    cost = torch.empty(S, P, dtype=torch.float64, device="cuda")
    w = torch.zeros(S, P, nmax + 1, dtype=torch.float64, device="cuda")
    grad = torch.zeros(S, P, nmax, dtype=torch.float64, device="cuda")
    for s in range(S):
        a, b, n = int(offs[s]), int(offs[s + 1]), int(N[s])
        step = max(1, int(2e8 // ((b - a) * (n + 1))))
        for p in range(0, P, step):
            c, x, gr = _cost64(om[a:b], er[a:b], ei[a:b], theta[s, p:p + step, :n], case["kind"])
            cost[s, p:p + step] = c
            w[s, p:p + step, :n + 1] = x
            if gr is not None:
                grad[s, p:p + step, :n] = gr
    if case["kind"] == "grad":
        return cost, grad
    return (cost, w) if case.get("weights") else cost
