"""Host-side check that the warp items of a central list fit the arrays made for them, for every number
of centrals the library accepts (include of the library's internal header, compiled for the host
with nvcc; no GPU).

A cell with v > 3 centrals gives ceil(v / (32 / L)) items, L the larger of lanes_per_central (at
most 4) and fill_lanes; one of 1 .. 3 centrals gives one.  The arrays hold one item per cell of the
grid and one per 8 ions."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include "ps_internal.cuh"
using namespace ps;
int main() {
  int bad = 0;
  const uint64_t want = kFillItems * 32ull;
  uint64_t n[64];
  int m = 0;
  for (uint64_t v : {0ull, 1ull, 2ull, 3ull, 31ull, 32ull, 33ull, 65536ull, 1ull << 20, 0xFFFFFFFEull}) n[m++] = v;
  for (uint64_t d : {2ull, 4ull, 8ull})
    for (uint64_t v : {want / d - 1, want / d, want / d + 1}) n[m++] = v;
  for (int s = 28; s < 32; ++s)  // sums and products of 32 bits would wrap here
    for (uint64_t v : {(1ull << s) - 1, 1ull << s, (1ull << s) + 1, (1ull << s) + want / 16}) n[m++] = v;
  for (int i = 0; i < m; ++i) {
    // the most lanes that still leave no more than `want` of them
    uint32_t L = 8;
    while (L > 1 && n[i] * L > want) L /= 2;
    if (fill_lanes((uint32_t)n[i]) != L) {
      printf("fill_lanes(%llu) = %u, not %u\n", (unsigned long long)n[i], fill_lanes((uint32_t)n[i]), L);
      ++bad;
    }
    // a list of n centrals in a grid made for n ions, the cells' remainders and light cells one item each
    const uint64_t lanes = fill_lanes((uint32_t)n[i]) > 4 ? fill_lanes((uint32_t)n[i]) : 4u;
    const uint64_t cells = n[i] / 8 > 65536 ? n[i] / 8 : 65536;
    const uint64_t items = n[i] / (32 / lanes) + (cells < n[i] ? cells : n[i]);
    if (items > cells + n[i] / 8 + 2) {
      printf("%llu centrals: %llu items\n", (unsigned long long)n[i], (unsigned long long)items);
      ++bad;
    }
  }
  // the lanes of the smallest items: a power of two, at most 16, that fits a warp
  for (uint32_t cnt = 1; cnt <= 3; ++cnt) {
    const uint32_t L = item_lanes(cnt);
    if ((L & (L - 1)) || L < 8 || L > 16 || cnt * L > 32) { printf("item_lanes(%u) = %u\n", cnt, L); ++bad; }
  }
  printf(bad ? "FAIL %d\n" : "OK\n", bad);
  return bad ? 1 : 0;
}
"""


def test_items_fit_their_arrays(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "bounds.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "bounds"
    subprocess.check_call([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "paper_2004_05188_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout
