"""Layouts whose blocks are not whole warps (csrc/launch.h, whole_warps): refused as host code
on the CPU, and a layout cache that names one is passed over, on the GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from oracle import dls, models

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_01928_gb300", "csrc")
BROKEN = [(4, 4), (1, 1), (3, 16), (5, 8), (33, 1), (2, 8), (64, 4), (256, 1), (1 << 30, 4), (0, 32), (32, 3),
          (32, 0), (4, -8), (1, 64)]
WHOLE = [(1, 32), (2, 16), (4, 8), (8, 16), (32, 1), (96, 1), (128, 1), (64, 2), (12, 8), (2, 32)]

HARNESS = r'''
#include <cstdio>
#include <cstdlib>
#include "launch.h"
int main(int c, char** v) {
  for (int i = 1; i + 1 < c; i += 2)
    std::printf("%d ", (int)debyefit::whole_warps(debyefit::Layout{std::atoi(v[i]), std::atoi(v[i + 1])}));
  return 0;
}
'''


def test_whole_warps(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "h.cu", tmp_path / "h"
    src.write_text(HARNESS)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o",
                        str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    args = [str(n) for l in BROKEN + WHOLE for n in l]
    out = subprocess.run([str(exe)] + args, capture_output=True, text=True, check=True).stdout.split()
    assert out == ["0"] * len(BROKEN) + ["1"] * len(WHOLE)


@pytest.mark.gpu
@pytest.mark.parametrize("line", ["64 1 4 4", "64 1 3 16", "64 1 1 1", "48 1 8 8", "1073741824 4 8 8"])
def test_cache_with_a_broken_layout_is_passed_over(line, tmp_path):
    torch = pytest.importorskip("torch")
    from paper_2109_01928_gb300 import debyefit as D
    b = W.mixed_batch(S=4, seed=3, P=32, K_range=(20, 60), N_range=(2, 4))
    re, im = models.synthesize(b)
    sp = D.make_spectra(b.offsets, b.omega, re, im, b.n_poles, b.lo, b.hi, device="cuda")
    th = W.population(b, 32, seed=2)
    theta = torch.as_tensor(th, device="cuda")
    path = str(tmp_path / "layouts")
    with D.Handle("mixed") as h:
        D.debye_autotune(h, sp, theta, cache_path=path)
    key, own = open(path).read().strip().split(" | ")
    open(path, "w").write(f"{key} | {line}\n")
    with D.Handle("mixed") as h:
        D.debye_autotune(h, sp, theta, cache_path=path)
        lines = open(path).read().strip().split("\n")
        assert len(lines) == 2 and lines[0].endswith(line)      # tuned anew, its own line added
        cb, ks, pcb, pks = (int(v) for v in lines[1].split(" | ")[1].split())
        assert cb % 32 == 0 and pcb * pks % 32 == 0
        out = D.debye_fit_batch(h, sp, P=32, iters=3, seed=1, polish_topk=3, polish_iters=4)
        cost = D.debye_eval_population(h, sp, theta).cpu().numpy()
        D.debye_sync(h)
    assert torch.isfinite(out["final_cost"]).all()
    for s in range(b.S):
        a, c = b.offsets[s], b.offsets[s + 1]
        ref, _ = dls.cost_population(b.omega[a:c], re[a:c], im[a:c], th[s, :, :int(b.n_poles[s])])
        assert np.max(np.abs(cost[s] - ref) / ref) <= 1e-5
