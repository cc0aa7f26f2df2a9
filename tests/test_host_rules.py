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


def _run(tmp_path, src):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no host compiler or CUDA headers")
    f = tmp_path / "t.cpp"
    f.write_text(src)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-O2", "-std=gnu++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
                    "/usr/local/cuda/include", "-o", exe, str(f)], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout


def test_product_tiles_fit_the_grid(tmp_path):
    n, bad = map(int, _run(tmp_path, GEMM).split())
    assert n > 10000 and bad == 0


def test_a_failed_allocation_leaves_the_projections(tmp_path):
    """Captured Lanczos loops hold the addresses of the projections: they may go only once their successors are
    there, and the loops with them."""
    rows = _run(tmp_path, PAIR).split("\n")
    assert rows[:3] == ["1 1 1 1", "0 1 1 0", "0 1 1 0"]
