"""The rules that choose between two forms of a search step (csrc/search.h): their lines, as host
code on the CPU, and the same bits from both forms, on the GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from oracle import models

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_01928_gb300", "csrc")


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    """rule(["expression", ...]): their values as integers."""
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("rules")

    def values(exprs):
        src, exe = d / "h.cu", d / "h"
        src.write_text('#include <cstdio>\n#include "launch.h"\n#include "search.h"\nusing namespace debyefit;\n'
                       'int main() {\n' + "".join(f'std::printf("%d ", (int)({e}));\n' for e in exprs) + "}\n")
        r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src),
                            "-o", str(exe)], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-2000:]
        return [int(v) for v in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()]
    return values


def test_swarm_step_goes_by_coordinates_per_spectrum(rule):
    cases = {(1, 64, 3): 1, (1, 64, 20): 1, (1, 128, 10): 1, (1, 129, 10): 0, (1, 80, 16): 1, (1, 81, 16): 0, (5, 77, 18): 1, (1, 77, 20): 0, (1, 1024, 1): 1, (1, 1024, 20): 0,
             (40, 128, 10): 1, (41, 131, 10): 1, (64, 200, 10): 1, (64, 205, 10): 0, (152, 243, 20): 1,
             (152, 244, 20): 0, (1024, 256, 12): 1, (1024, 1024, 20): 1, (1024, 1025, 1): 0, (1 << 20, 1025, 20): 0}
    assert rule([f"pso_step_fused({s}ll, {p}, {n})" for s, p, n in cases]) == list(cases.values())


def test_polish_round_goes_by_trials_and_poles(rule):
    # (lines, trials, poles, longest spectrum, precision) on 152 SMs
    cases = {(8, 19, 3, 50, "MIXED"): 1, (8, 8, 3, 50, "MIXED"): 0, (8, 9, 3, 50, "MIXED"): 1, (8, 32, 3, 50, "MIXED"): 1,
             (8, 33, 3, 50, "MIXED"): 0, (8, 0, 3, 50, "MIXED"): 0, (8, 19, 20, 1 << 20, "MIXED"): 1,
             (512, 19, 20, 1 << 30, "MIXED"): 1, (1024, 19, 20, 4000, "MIXED"): 0, (1024, 19, 20, 1000, "MIXED"): 1, (2048, 19, 8, 1000, "MIXED"): 1, (2048, 19, 8, 1200, "MIXED"): 0,
             (1496, 19, 16, 180, "MIXED"): 1, (2048, 19, 12, 1000, "MIXED"): 0, (2049, 19, 1, 2, "MIXED"): 0,
             (2048, 19, 14, 4000, "MIXED_TABLE"): 1, (2048, 19, 15, 50, "MIXED_TABLE"): 0,
             (2049, 19, 1, 50, "MIXED_TABLE"): 0, (512, 19, 20, 4000, "FP64"): 1, (1024, 19, 12, 400, "FP64"): 1,
             (1024, 19, 13, 400, "FP64"): 0, (2048, 19, 5, 50, "FP64"): 1, (2048, 19, 6, 50, "FP64_SUMS"): 0,
             (1 << 40, 32, 20, 1 << 30, "FP64_SUMS"): 0}
    assert rule([f"polish_one_round({l}ll, {t}, {n}, {k}ll, DEBYE_PREC_{p}, 152)"
                 for l, t, n, k, p in cases]) == list(cases.values())


@pytest.mark.gpu
@pytest.mark.parametrize("P,N", [(257, 5), (300, 7), (1024, 2)])
def test_swarm_steps_of_both_forms_agree(P, N):
    # the first spectrum of a batch large enough for the step in one kernel, and alone, where
    # it takes two: the same layout and solve, so the same bits
    torch = pytest.importorskip("torch")
    from paper_2109_01928_gb300 import debyefit as D
    S = -(-P * N // 32)
    b = W.mixed_batch(S=S, seed=41, P=P, K_range=(24, 24), N_range=(N, N))
    re, im = models.synthesize(b)
    traces = []
    for n in (S, 1):
        k = int(b.offsets[n])
        sp = D.make_spectra(b.offsets[:n + 1], b.omega[:k], re[:k], im[:k], b.n_poles[:n], b.lo[:n], b.hi[:n], device="cuda")
        with D.Handle("mixed", cands_per_block=64, lanes_per_candidate=2, solve_lanes=1) as h:
            out = D.debye_fit_batch(h, sp, P=P, iters=6, seed=5, polish_topk=0, trace=True)
            D.debye_sync(h)
        traces.append((out["trace"][0].cpu().numpy(), out["tau"][0].cpu().numpy()))
    assert np.isfinite(traces[0][0]).all()
    for a, c in zip(*traces):
        assert np.array_equal(a, c)
