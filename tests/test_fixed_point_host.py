"""The fixed-point contractions (csrc/fixed.cuh) in their host form: one element of Hbar, the
stages of csrc/hbar_fx.cu in order, beside the chain of folded FP64 contractions that it
stands for, both against extended precision with the same tables.

The vectors go from dense ones to ones that fall off by 69 e-folds along the element or have
one large entry: the entries of an element share one exponent, so small ones are where a
fixed-point form can lose bits.  The bounds: the 2-norm error is no larger than the FP64
chain's, and no larger than one rounding (2^-53) of the sums of magnitudes behind the results."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_13130_gb300", "csrc")

SOURCE = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>
#include "fixed.cuh"
#include "tdks_internal.h"
using namespace tdks;
typedef long double ld;
template <class T> using Vec = std::vector<T>;

template <class T> Vec<T> fold(const Vec<T>& M, int n) {      // the layout of tdks_internal.h
  const int h = n / 2;
  Vec<T> f(2 * h * h + 2 * h + 1, 0);
  for (int q = 0; q < h; ++q)
    for (int i = 0; i < h; ++i) {
      f[q * h + i] = (M[q * n + i] + M[q * n + n - 1 - i]) / 2;
      f[h * h + q * h + i] = (M[q * n + i] - M[q * n + n - 1 - i]) / 2;
    }
  if (n & 1) {
    for (int q = 0; q < h; ++q) f[2 * h * h + q] = M[q * n + h];
    for (int i = 0; i <= h; ++i) f[2 * h * h + h + i] = M[h * n + i];
  }
  return f;
}
template <class T> Vec<T> transpose(const Vec<T>& M, int n) {
  Vec<T> t(M);
  for (int a = 0; a < n; ++a) for (int b = 0; b < n; ++b) t[b * n + a] = M[a * n + b];
  return t;
}
int stride(int n, int ax) { return ax == 0 ? 1 : ax == 1 ? n : n * n; }
template <int N, class F> void lines(int ax, F f) {
  const int st = stride(N, ax);
  for (int i = 0; i < N * N * N; ++i) if (i / st % N == 0) f(i, st);
}
template <int N> Vec<ld> dense(const Vec<ld>& M, const Vec<ld>& x, int ax) {
  Vec<ld> y(x.size(), 0);
  lines<N>(ax, [&](int i, int st) { for (int a = 0; a < N; ++a) for (int b = 0; b < N; ++b) y[i + a * st] += M[a * N + b] * x[i + b * st]; });
  return y;
}
// (B'^T)^(x)3 [sum_d cd K'_d + J V] B'^(x)3 y; U and R by the way
template <int N> Vec<ld> exact(const Vec<ld>& B, const Vec<ld>& K, const Vec<double>& JV, const double* cd, const Vec<double>& y, bool mag, ld* ur) {
  auto m = [&](Vec<ld> M) { if (mag) for (ld& v : M) v = fabsl(v); return M; };
  Vec<ld> x(y.begin(), y.end());
  x = m(x);
  for (int ax = 2; ax >= 0; --ax) x = dense<N>(m(B), x, ax);
  Vec<ld> r(x.size());
  for (size_t i = 0; i < x.size(); ++i) r[i] = (mag ? fabsl(JV[i]) : (ld)JV[i]) * x[i];
  for (int ax = 0; ax < 3; ++ax) {
    const Vec<ld> t = dense<N>(m(K), x, ax);
    for (size_t i = 0; i < x.size(); ++i) r[i] += cd[ax] * t[i];
  }
  *ur = 0;
  for (size_t i = 0; i < x.size(); ++i) *ur += x[i] * r[i];
  for (int ax = 2; ax >= 0; --ax) r = dense<N>(transpose(m(B), N), r, ax);
  return r;
}
template <int N> void apply64(const Vec<double>& t, Vec<double>& x, int ax) {
  constexpr int h = N / 2;
  lines<N>(ax, [&](int i0, int st) {
    double e[N], o[N], y[N];
    for (int i = 0; i < h; ++i) e[i] = x[i0 + i * st] + x[i0 + (N - 1 - i) * st], o[i] = x[i0 + i * st] - x[i0 + (N - 1 - i) * st];
    const double mid = x[i0 + h * st];
    for (int q = 0; q < h; ++q) {
      double a = 0, b = 0;
      for (int i = 0; i < h; ++i) a = fma(t[q * h + i], e[i], a), b = fma(t[h * h + q * h + i], o[i], b);
      if (N & 1) a = fma(t[2 * h * h + q], mid, a);
      y[q] = a + b, y[N - 1 - q] = a - b;
    }
    if (N & 1) {
      y[h] = t[2 * h * h + 2 * h] * mid;
      for (int i = 0; i < h; ++i) y[h] = fma(t[2 * h * h + h + i], e[i], y[h]);
    }
    for (int q = 0; q < N; ++q) x[i0 + q * st] = y[q];
  });
}
template <int N> Vec<double> chain64(const Tables1D& T, const Vec<double>& JV, const double* cd, const Vec<double>& y) {
  const Vec<double> B = fold(T.B, N), BT = fold(transpose(T.B, N), N), K = fold(T.Kq, N);
  Vec<double> u = y, r(y.size());
  for (int ax = 2; ax >= 0; --ax) apply64<N>(B, u, ax);
  const auto& w = T.omega;
  for (int i = 0; i < N * N * N; ++i) r[i] = JV[i] * (w[i / N % N] * w[i / N / N]) * w[i % N] * u[i];
  for (int ax = 0; ax < 3; ++ax) {
    Vec<double> t = u;
    apply64<N>(K, t, ax);
    for (int i = 0; i < N * N * N; ++i) {
      const double wl = ax == 0 ? w[i / N % N] * w[i / N / N] : ax == 1 ? w[i % N] * w[i / N / N] : w[i % N] * w[i / N % N];
      r[i] = fma(cd[ax] * wl, t[i], r[i]);
    }
  }
  for (int ax = 2; ax >= 0; --ax) apply64<N>(BT, r, ax);
  return r;
}
struct Op { Vec<FxC> c; Vec<float> k; };
template <int N, class F> Op table(F coef) {
  Op o;
  for (int i = 0; i < FxOp<N>::CS; ++i) o.c.push_back(fx_coef(coef(i)));
  for (int i = 0; i < FxOp<N>::KS; ++i) o.k.push_back(fx_tail_const<N>([&](int j) { return o.c[j]; }, i));
  return o;
}
struct Val { Vec<long long> v; Vec<float> f; };
bool range_ok = true;
template <int N> void apply(const Op& o, Val& x, int ax) {
  lines<N>(ax, [&](int i0, int st) {
    long long v[N];
    float f[N];
    for (int i = 0; i < N; ++i) {
      v[i] = x.v[i0 + i * st], f[i] = x.f[i0 + i * st];
      range_ok &= std::llabs(v[i]) < (1ll << 55) + (1 << 23) && fabsf(f[i]) < 8;
    }
    fx_apply<N>([&](int i) { return o.c[i]; }, [&](int i) { return o.k[i]; }, v, f,
                [&](int q, long long a, float b) { x.v[i0 + q * st] = a, x.f[i0 + q * st] = b; });
  });
}
int field(double x) {   // biased exponent
  uint64_t b;
  memcpy(&b, &x, 8);
  return (int)(b >> 52 & 0x7ff);
}
template <int N> Vec<double> chain_fx(const Tables1D& T, const Vec<double>& JV, const double* cd, const Vec<double>& y, ld* ur) {
  const int n = N * N * N;
  const Vec<ld> fB = fold(T.Bw, N), fBT = fold(transpose(T.Bw, N), N), fK = fold(T.Kw, N);
  const Op B = table<N>([&](int i) { return llrintl(ldexpl(fB[i], 63)); }), BT = table<N>([&](int i) { return llrintl(ldexpl(fBT[i], 63)); });
  double vm = 0, ym = 0;
  for (double v : JV) vm = fmax(vm, fabs(v));
  for (double v : y) ym = fmax(ym, fabs(v));
  const double bound = (T.kw_inf * (cd[0] + cd[1] + cd[2]) + vm * (1 + 0x1p-20)) * 1.0000001;
  const int er = field(bound) - 1022, eb = field(ym);
  const double scale = ldexp(1.0, 63 - er);
  Val a{Vec<long long>(n), Vec<float>(n, 0)};
  for (int i = 0; i < n; ++i) {
    uint64_t b;
    memcpy(&b, &y[i], 8);
    a.v[i] = fx_from_bits((unsigned)(b >> 32), (unsigned)b, eb, a.f[i]);
  }
  apply<N>(B, a, 2);
  apply<N>(B, a, 1);
  unsigned big = 0;
  for (long long v : a.v) big |= fx_magnitude(v);
  const int up = fx_free_bits(big);
  for (int i = 0; i < n; ++i) fx_raise(a.v[i], a.f[i], up);
  apply<N>(B, a, 0);
  Val r = a;
  for (int ax = 0; ax < 3; ++ax) {
    Val t = a;
    apply<N>(table<N>([&](int i) { return fx_scaled(cd[ax], (double)fK[i], (double)(fK[i] - (double)fK[i]), scale); }), t, ax);
    for (int i = 0; i < n; ++i) {
      if (ax == 0) {
        const FxC w = fx_coef(llrint(JV[i] * scale));
        const FxV q = fx_operand(a.v[i] + kFxHalf, a.f[i]);
        FxDot d;
        d.term(w, q);
        d.close(fmaf(w.cl, -1.5f, -1.5f));
        d.top(w, q);
        r.v[i] = t.v[i] + d.hi, r.f[i] = t.f[i] + d.f;
      } else {
        r.v[i] += t.v[i], r.f[i] += t.f[i];
      }
    }
  }
  *ur = 0;
  lines<N>(2, [&](int i0, int st) {
    FxInner s;
    for (int i = 0; i < N; ++i) s.add(a.v[i0 + i * st], a.f[i0 + i * st], r.v[i0 + i * st], r.f[i0 + i * st]);
    *ur += ldexpl((ld)s.dh, 64) + ldexpl((ld)s.dm + (ld)s.da, 32) + ldexpl((ld)s.dl, 10);
  });
  *ur = ldexpl(*ur, er + 7 - 2 * (kFxBits - eb + 1022 + up));
  for (int ax = 2; ax >= 0; --ax) apply<N>(BT, r, ax);
  Vec<double> out(n);
  for (int i = 0; i < n; ++i) out[i] = (double)ldexpl((ld)r.v[i] + (ld)r.f[i], er + 7 - kFxBits + eb - 1022 - up);
  return out;
}
template <int N> void all() {
  const Tables1D T = tdks_build_tables(N - 1, N);
  const int n = N * N * N;
  std::mt19937_64 g(5 + N);
  auto uni = [&] { return (double)(int64_t)g() * 0x1p-63; };
  for (int pot = 0; pot < 2; ++pot) {
    Vec<double> JV(n), y(n);
    for (double& v : JV) v = pot ? -3 + uni() : -200 * exp(4 * uni());
    const double cd[3] = {0.5, 0.4375, 0.53125};
    for (int kind = 0; kind < 14; ++kind) {
      const double s[] = {0, 2, 8, 20, 40, 1e-2, 1e-4, 1e-8};
      for (int i = 0; i < n; ++i) {
        const double a = 1 + T.xi[i % N], b = 1 + T.xi[i / N % N], c = 1 + T.xi[i / N / N];
        const int k = kind / 2;
        y[i] = (kind % 2 || k == 0 ? uni() : 1.0) * (k < 5 ? exp(-s[k] * sqrt(a * a + b * b + c * c) / 2) : i ? s[k] : 1.0);
      }
      ld ur, um, uf;
      const Vec<ld> ex = exact<N>(T.Bw, T.Kw, JV, cd, y, false, &ur), mg = exact<N>(T.Bw, T.Kw, JV, cd, y, true, &um);
      const Vec<double> d = chain64<N>(T, JV, cd, y), f = chain_fx<N>(T, JV, cd, y, &uf);
      ld e64 = 0, efx = 0, m = 0, sum = 0;
      for (int i = 0; i < n; ++i) e64 += (d[i] - ex[i]) * (d[i] - ex[i]), efx += (f[i] - ex[i]) * (f[i] - ex[i]), m += mg[i] * mg[i], sum += ex[i] * ex[i];
      printf("%d %d %d %.3e %.3e %.3e %.3e %d\n", N - 1, pot, kind, (double)sqrtl(e64 / sum), (double)sqrtl(efx / sum), (double)sqrtl(efx / m), (double)(fabsl(uf - ur) / um), (int)range_ok);
    }
  }
}
int main() { all<2>(); all<3>(); all<4>(); all<5>(); all<6>(); all<7>(); all<8>(); all<9>(); }
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no host compiler or CUDA headers")
    d = tmp_path_factory.mktemp("fx")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-O1", "-std=gnu++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
                    "/usr/local/cuda/include", "-o", str(d / "t"), str(d / "t.cpp"), os.path.join(CSRC, "tables.cpp")],
                   check=True)
    out = subprocess.run([str(d / "t")], check=True, capture_output=True, text=True).stdout
    return [[float(x) for x in l.split()] for l in out.splitlines()]


@pytest.mark.parametrize("p", range(1, 9))
def test_element_operator_is_as_accurate_as_fp64(rows, p):
    mine = [r for r in rows if r[0] == p]
    assert len(mine) == 28
    for _, pot, kind, e64, efx, emag, _, ok in mine:
        assert ok, "a value left its range"
        assert efx <= e64 and emag <= 2.0 ** -53, (pot, kind, e64, efx, emag)


@pytest.mark.parametrize("p", range(1, 9))
def test_energy_of_an_element(rows, p):
    """u . r, the element's part of a Lanczos alpha: integers and tails, within 2^-56 of the sum of magnitudes (an FP64
    sum rounds every term to 2^-53)."""
    for _, pot, kind, _, _, _, eur, _ in (r for r in rows if r[0] == p):
        assert eur <= 2.0 ** -56, (pot, kind, eur)
