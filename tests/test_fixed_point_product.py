"""The fixed-point products of the Poisson preconditioner (FxSum in csrc/fixed.cuh, the arithmetic
of k_gemm_fx in csrc/poisson.cu) in their host form, beside FP64 chains, both against 113-bit
arithmetic: the eigenvector matrices of uniform and graded axes of 3 to 255 interior nodes, both
ways, times columns that are dense, smooth, over 12 and 30 decades, that fall off by up to 80
e-folds, or have one large entry."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_13130_gb300", "csrc")

SOURCE = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>
#include "fixed.cuh"
#include "tdks_internal.h"
using namespace tdks;
int field(double x) {
  uint64_t b;
  memcpy(&b, &x, 8);
  return (int)(b >> 52 & 0x7ff);
}
FxV factor(double x, int eb) {
  uint64_t b;
  memcpy(&b, &x, 8);
  return fx_factor((unsigned)(b >> 32), (unsigned)b, eb);
}
// a sum and what its additions leave: 106 bits
struct Sum {
  double h = 0, l = 0;
  void add(double x) { const double s = h + x, v = s - h; l += (h - (s - v)) + (x - v); h = s; }
};
int main() {
  std::mt19937_64 g(11);
  auto uni = [&] { return (double)(int64_t)g() * 0x1p-63; };
  const struct { int p, n; double ratio; } axes[] = {
      {2, 2, 1}, {1, 4, 1.25}, {2, 3, 1.25}, {2, 4, 1.25}, {4, 2, 1}, {4, 4, 1.25}, {8, 2, 1.25}, {1, 17, 1.25}, {6, 3, 1}, {4, 6, 1},
      {8, 4, 1}, {3, 11, 1.5}, {2, 17, 1.25}, {6, 14, 1}, {6, 16, 1}, {5, 20, 1.25}, {8, 12, 2}, {4, 50, 1}, {8, 32, 1.05}, {8, 32, 1}};
  for (const auto& m : axes) {
    std::vector<double> br(m.n + 1, 0.0), S, lam;
    for (int e = 0; e < m.n; ++e) br[e + 1] = br[e] + pow(m.ratio, fabs(e - 0.5 * (m.n - 1)));
    for (double& v : br) v *= 2.0 * m.n / br[m.n];
    tdks_fdm_axis(tdks_build_tables(m.p, m.p + 1), m.p, br.data(), m.n, S, lam);
    const int K = m.n * m.p - 1;
    for (int kind = 0; kind < 12; ++kind)
      for (int back = 0; back < 2; ++back) {
        std::vector<double> b(K);
        const int at = (int)(fabs(uni()) * (K - 1));
        const double st = 10 + 70 * fabs(uni());
        for (int j = 0; j < K; ++j) {
          const double r = uni(), x = (double)j / K, d = fabs(j - at) / K;
          b[j] = kind == 0 ? r : kind == 1 ? exp(-pow((x - 0.5) * 6, 2)) : kind == 2 ? r * pow(10, -12 * fabs(uni()))
                 : kind == 3 ? exp(-st * x) : kind == 4 ? exp(-st * (1 - x)) : kind == 5 ? (j == at) + 1e-9 * r
                 : kind == 6 ? exp(-st * d) : kind == 7 ? r * exp(-st * d) : kind == 8 ? r / (1 + lam[j])
                 : kind == 9 ? r * exp(-st * x) : kind == 10 ? (j == at) + 1e-4 * r : r * pow(10, -30 * fabs(uni()));
        }
        double e64 = 0, efx = 0, sum = 0;
        int bad = 0;
        for (int i = 0; i < K; ++i) {
          const double* a = back ? &S[(size_t)i * K] : &S[i];
          const int sa = back ? 1 : K;
          int ea = 64, eb = 64;
          for (int k = 0; k < K; ++k) ea = std::max(ea, field(a[k * sa])), eb = std::max(eb, field(b[k]));
          Sum x;
          FxSum f;
          double d = 0;
          for (int k = 0; k < K; ++k) {
            const double p = a[k * sa] * b[k];
            x.add(p);
            x.add(fma(a[k * sa], b[k], -p));
            d = fma(a[k * sa], b[k], d);
            const FxV u = factor(a[k * sa], ea), w = factor(b[k], eb);
            bad += std::abs(u.h) > 1 << 26 || std::abs(w.h) > 1 << 26;
            f.add(u.h, u.l, u.g - 1.5f, w.h, w.l, w.g - 1.5f);
            if (k % 16 == 15) f.carry();
          }
          int s;
          const long long v = f.value(s);
          bad += s < 1 || s > 20 || std::llabs(v) >= 1ll << 62;
          const double y = ldexp((double)v, 64 - s + (ea - 1022 - kFxPBits) + (eb - 1022 - kFxPBits));
          e64 += pow((d - x.h) - x.l, 2), efx += pow((y - x.h) - x.l, 2), sum += x.h * x.h;
        }
        printf("%d %d %.3e %.3e %d\n", K, kind, sqrt(e64 / sum), sqrt(efx / sum), bad);
      }
  }
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no host compiler or CUDA headers")
    d = tmp_path_factory.mktemp("fxp")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-O1", "-std=gnu++17", "-ffp-contract=off", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", "/usr/local/cuda/include", "-o", str(d / "t"), str(d / "t.cpp"),
                    os.path.join(CSRC, "tables.cpp"), os.path.join(CSRC, "fdm.cpp")], check=True)
    out = subprocess.run([str(d / "t")], check=True, capture_output=True, text=True).stdout
    return [[float(x) for x in l.split()] for l in out.splitlines()]


def test_products_are_as_accurate_as_fp64(rows):
    """In the 2-norm no further off than the FP64 chain, or than one rounding of the results (2^-53), which a chain of
    few terms may stay below."""
    assert len(rows) == 20 * 12 * 2
    for K, kind, e64, efx, bad in rows:
        assert bad == 0, (K, kind)
        assert efx <= max(e64, 2.0 ** -53), (K, kind, e64, efx)
