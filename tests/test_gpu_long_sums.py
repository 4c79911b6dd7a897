"""The end of the column-sum pass (csrc/eval.cuh, sums_write) on the sums of very long spectra,
against the FP64 forms: S and the derivative sum U carry a bias of 1 per lane, whose removal
FP32 holds exactly only below 2^24. Bit for bit, on both sides of 2^24."""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_01928_gb300", "csrc")

SRC = r"""
#include "common.cuh"
#include "eval.cuh"
#include <cstdio>
using namespace debyefit;
__device__ int bad[4];
__device__ double bits_of(ff a, ff b) { return fabs((double)a.h - (double)b.h) + fabs((double)a.l - (double)b.l); }
__global__ void check(int ks, double* x, double* G) {   // one thread: x[1], G[4]
  constexpr double LN10 = 2.302585092994046;
  const double tau = 3e-9;
  // whole numbers around 2^24 and 2^25, odd ones where FP32 has them, and small sums
  const float hs[] = {(float)ks, 33.f, 700.5f, 0x1p23f + 1.f, 0x1p24f - 1.f, 0x1p24f, 0x1p24f + 2.f, 0x1p24f + 6.f,
                      0x1p25f, 0x1p25f + 4.f, 0x1p28f + 32.f, 0x1p30f};
  const float ls[] = {0.f, 0.3f, -0.7f, 1.f, 2.5f, -1e-7f};
  for (float h : hs)
    for (float l : ls) {
      PoleSums<true> s;
      s.sh = s.uh = h;
      s.sl = s.ul = l;
      s.ah = 7.f, s.al = 1e-8f, s.ch = 5e9f, s.cl = 100.f;
      s.vh = 2.f, s.vl = -1e-9f, s.wh = 1e9f, s.wl = 3.f;
      const double S = ((double)h - (double)ks) + (double)l;
      const double D = -2.0 * LN10 * S;
      x[0] = tau;
      sums_write<true>(x, G, 1, s, ks, true);
      if (G[0] != S) ++bad[0];
      if (G[2] != D) ++bad[1];
      x[0] = tau;
      sums_write<true>(x, G, 1, s, ks, false);
      const ff a = load_ff(G, 0), d = load_ff(G, 2), A = ff_of(S), E = ff_of(D);
      if (bits_of(a, A) != 0.0) ++bad[2];
      if (bits_of(d, E) != 0.0) ++bad[3];
    }
}
int main(int, char** v) {
  double* p;
  cudaMalloc(&p, sizeof(double) * 5);
  check<<<1, 1>>>(std::atoi(v[1]), p, p + 1);
  int h[4];
  const cudaError_t e = cudaMemcpyFromSymbol(h, bad, sizeof(h));
  if (e != cudaSuccess) { std::printf("%s\n", cudaGetErrorString(e)); return 2; }
  std::printf("%d %d %d %d\n", h[0], h[1], h[2], h[3]);
  return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("long")
    src, out = d / "long.cu", d / "long"
    src.write_text("#include <cstdlib>\n" + SRC)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o",
                        str(out)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return str(out)


@pytest.mark.parametrize("ks", [1, 2, 4, 32])
def test_bias_of_long_sums(exe, ks):
    r = subprocess.run([exe, str(ks)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert r.stdout.split() == ["0", "0", "0", "0"]     # S, D in FP64; S, D in float-float
