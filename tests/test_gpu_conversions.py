"""The integer conversions between FP64 and float-float and the reciprocal (csrc/common.cuh)
and the table's segment lookup (csrc/tables.cu) against the plain FP64 forms, bit for bit (a zero low part
may differ in its sign), over random bit patterns and the edges of their ranges: powers of
two and their neighbours, ties, carries into the exponent, zeros, subnormal and huge
values, infinities and NaN."""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2109_01928_gb300", "csrc")

SRC = r"""
#include "tables.cu"
#include <cstdio>
using namespace debyefit;
__device__ unsigned long long bad[6];
__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b) || a == b || (isnan(a) && isnan(b)); }
__device__ bool same(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b) || (isnan(a) && isnan(b)); }
__device__ void check_double(double v) {
  const float h = __double2float_rn(v), l = __double2float_rn(v - (double)h);
  const ff r = ff_of(v);
  if (!same(r.h, h) || !same(r.l, l)) atomicAdd(&bad[0], 1ull);
  for (int ns = 1; ns <= 1000; ns = ns * 10) {
    const int g = (v >= 0.0 && v <= (double)ns) ? min((int)v, ns - 1) : -1;
    if (tab_segment(v, ns) != g) atomicAdd(&bad[3], 1ull);
  }
}
__device__ void check_pair(float a, float b) {   // normalised by two_sum
  if (!same(dbl_of(a), (double)a) || !same(dbl_of(b), (double)b)) atomicAdd(&bad[1], 1ull);
  ff f;
  two_sum(a, b, f.h, f.l);
  if (!isfinite(f.h)) return;
  const double v = (double)f.h + (double)f.l;
  const ff p{__double2float_rn(v), __double2float_rn(v - (double)__double2float_rn(v))};
  const ff r = ff_round53(f);
  if (!same(r.h, p.h) || !same(r.l, p.l)) atomicAdd(&bad[2], 1ull);
}
__global__ void check(int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint64_t k = splitmix64(i), k2 = splitmix64(k);
    // every exponent; fractions random, or all zeros / ones, or near the rounding ties
    uint64_t frac = k & 0xfffffffffffffull;
    switch (i % 8) {
      case 1: frac = 0; break;
      case 2: frac = 0xfffffffffffffull; break;
      case 3: frac = (frac & ~0x1fffffffull) | 0x10000000ull; break;
      case 4: frac = (frac & ~0x1fffffffull) | 0x0fffffffull; break;
      case 5: frac = (frac & ~0x1fffffffull) | 0x10000001ull; break;
      case 6: frac = 0xfffffe0000000ull | (frac & 0x1fffffffull); break;
      case 7: frac &= ~0x1fffffffull; break;
    }
    const uint64_t e = (i & 8) ? 1023 - 90 + (k2 >> 8) % 230 : (k2 >> 8) % 2048;
    check_double(__longlong_as_double((long long)((k2 & 1) << 63 | e << 52 | frac)));
    check_double((double)((k2 >> 3) % 2100) + ((i & 16) ? 0.0 : (double)(k % 1000) * 1e-3));
    check_double(-(double)(i % 3));
    const uint32_t ha = (uint32_t)k, hb = (uint32_t)(k2 >> 32);
    check_pair(__uint_as_float(ha), __uint_as_float(hb));
    // a low part 24 to 60 binades below, at a power of two or not
    const float a = __uint_as_float((ha & 0x80000000u) | (64u + (ha >> 8) % 180u) << 23 | ((i & 32) ? 0u : ha & 0x7fffffu));
    const float b = __uint_as_float((hb & 0x807fffffu) | ((__float_as_uint(a) >> 23 & 0xffu) - 23u - (hb >> 24) % 37u) << 23);
    check_pair(a, b);
    check_pair(a, __uint_as_float(__float_as_uint(b) & 0xffff8000u));
    check_pair(a, 0.f);
    // denominators 1 + x^2: any binade, all-ones and near-power fractions, and just above 1
    const uint64_t ed = 1023 + (k2 >> 8) % ((i & 64) ? 1025 : 72);
    const double dd = (i & 128) ? 1.0 + ldexp((double)(k >> 11), -53 - (int)(k2 % 60))
                               : __longlong_as_double((long long)(ed << 52 | frac));
    if (!same(rcp_ge1(dd), 1.0 / dd)) atomicAdd(&bad[5], 1ull);
    const double dn = __longlong_as_double((long long)((ed << 52) + (long long)(k % 4096) - 2048));
    if (dn >= 1.0 && !same(rcp_ge1(dn), 1.0 / dn)) atomicAdd(&bad[5], 1ull);
    if (dbl_of_int(1 + i % 2001) != (double)(1 + i % 2001)) atomicAdd(&bad[4], 1ull);
    const int m = (int)(k >> 34);   // below 2^30
    const ff c = ff_of_int(m), d = ff_of((double)m);
    if (!same(c.h, d.h) || !same(c.l, d.l)) atomicAdd(&bad[4], 1ull);
  }
}
int main() {
  check<<<304, 256>>>(1 << 22);
  unsigned long long h[6];
  if (cudaMemcpyFromSymbol(h, bad, sizeof(h)) != cudaSuccess) return 1;
  printf("%llu %llu %llu %llu %llu %llu\n", h[0], h[1], h[2], h[3], h[4], h[5]);
  return 0;
}
"""


def test_integer_conversions_match_fp64(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, exe = tmp_path / "conv.cu", tmp_path / "conv"
    src.write_text(SRC)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I", CSRC, "-o",
                    str(exe), str(src)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["0"] * 6, dict(zip(("ff_of", "dbl_of", "ff_round53", "tab_segment", "integers", "rcp_ge1"), out))
