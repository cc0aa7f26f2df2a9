"""Host-side rules of the CUDA library (csrc/tdks_internal.h), compiled with the host compiler."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_13130_gb300", "csrc")

GEMM = r"""
#include <cstdio>
#include "tdks_internal.h"
int main() {
  // the products of the fast diagonalization: axes of at most 1024 nodes each
  const int ax[] = {1, 2, 3, 4, 7, 15, 16, 17, 31, 33, 64, 83, 100, 255, 256, 300, 1000, 1008, 1009, 1023, 1024};
  long long bad = 0, n = 0;
  for (int x : ax) for (int y : ax) for (int z : ax) {
    const long long M[3] = {(long long)y * z, y, z}, N[3] = {x, x, (long long)x * y}, B[3] = {1, z, 1};
    for (int d = 0; d < 3; ++d, ++n) {
      const int t = gemm_tile(M[d], N[d], B[d]);
      bad += (t != 16 && t != 32 && t != 64) || (M[d] + t - 1) / t > 65535 || B[d] > 65535;
    }
  }
  printf("%lld %lld\n", n, bad);
}
"""

PAIR = r"""
#include <cstdio>
#include <set>
#include "tdks_internal.h"
// projections replaced by larger ones: the allocation that fails (0: none), what is left after it
int main() {
  for (int fail = 0; fail < 3; ++fail) {
    static int heap[8];
    std::set<int*> live{heap, heap + 1};
    int *a = heap, *b = heap + 1, calls = 0, dropped = 0;
    const auto alloc = [&](size_t) -> int* {
      if (++calls == fail) return nullptr;
      live.insert(heap + 1 + calls);
      return heap + 1 + calls;
    };
    const bool ok = replace_pair(a, 5, b, 6, alloc, [&](int* p) { live.erase(p); },
                                 [&] { dropped += live.count(heap) && live.count(heap + 1); });
    const bool kept = a == heap && b == heap + 1, fresh = a == heap + 2 && b == heap + 3;
    printf("%d %d %d %d\n", (int)ok, fail ? kept : fresh, (int)(live == std::set<int*>{a, b}), dropped);
  }
}
"""

FOLD = r"""
#include <cmath>
#include <cstdio>
#include "tdks_internal.h"
typedef long double ld;
ld legendre(int p, ld x, ld* below) {
  ld a = 1, b = x;
  for (int k = 1; k < p; ++k) { const ld c = ((2 * k + 1) * x * b - k * a) / (k + 1); a = b; b = c; }
  *below = a;
  return b;
}
int main() {
  for (int p = 1; p <= 8; ++p) {
    // the 1-D stiffness from the closed form of differentiation at the GLL nodes and the GLL rule (exact for it)
    const int n = p + 1, h = n / 2;
    ld x[9], L[9], d[9][9], K[9][9] = {}, below;
    for (int i = 0; i < n; ++i) {
      x[i] = i == 0 ? -1 : i == p ? 1 : -cosl(acosl(-1.0L) * i / p);
      for (int it = 0; it < 50 && i > 0 && i < p; ++it) {
        const ld v = legendre(p, x[i], &below);
        x[i] -= (x[i] * v - below) / (n * v);
      }
    }
    for (int i = 0; i < h; ++i) x[p - i] = -x[i];
    if (n % 2) x[h] = 0;
    for (int i = 0; i < n; ++i) L[i] = legendre(p, x[i], &below);
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j)
        d[i][j] = i != j ? L[i] / (L[j] * (x[i] - x[j])) : i == 0 ? -p * n / 4.0L : i == p ? p * n / 4.0L : 0;
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j)
        for (int k = 0; k < n; ++k) K[i][j] += 2 / (p * n * L[k] * L[k]) * d[k][i] * d[k][j];
    const Tables1D t = tdks_build_tables(p, n);
    ld worst = 0;
    for (int q = 0; q < h; ++q)
      for (int i = 0; i < h; ++i)
        for (int k = 0; k < 2; ++k) {
          const ld e = 0.5L * (K[q][i] + (k ? -1 : 1) * K[q][p - i]);
          worst = fmaxl(worst, (fabsl(t.csK1[k * h * h + q * h + i] - e) - 1e-17L) / fabsl(e));
        }
    printf("%d %.4Lf\n", p, worst * 0x1p53L);
  }
}
"""


def _run(tmp_path, src, *more):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no host compiler or CUDA headers")
    f = tmp_path / "t.cpp"
    f.write_text(src)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-O2", "-std=gnu++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
                    "/usr/local/cuda/include", "-o", exe, str(f), *more], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout


def test_product_tiles_fit_the_grid(tmp_path):
    n, bad = map(int, _run(tmp_path, GEMM).split())
    assert n > 10000 and bad == 0


def test_a_failed_allocation_leaves_the_projections(tmp_path):
    """Captured Lanczos loops hold the addresses of the projections: they may go only once their successors are
    there, and the loops with them."""
    rows = _run(tmp_path, PAIR).split("\n")
    assert rows[:3] == ["1 1 1 1", "0 1 1 0", "0 1 1 0"]


def test_folded_stiffness_is_rounded_once(tmp_path):
    """Entries within half a unit of the exact ones, 2^-53 of themselves (a constant has no stiffness, and what the
    rounding leaves of it is amplified in the potential); the reference's own error is below 1e-17."""
    for line in _run(tmp_path, FOLD, os.path.join(CSRC, "tables.cpp")).splitlines():
        p, worst = line.split()
        assert float(worst) <= 1.0, (p, worst)
