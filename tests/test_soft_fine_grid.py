"""Host check of the smoothed RDF's fine grid (include of the library's internal header, compiled for the host
with nvcc): over ranges from a few to ten thousand sigma the bins fit, the width is at most sigma / 40 where the
bins allow it, and every bin centre is a float32 number."""
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
  for (double sig = 1e-4; sig < 50.0; sig *= 1.0371)
    for (double ratio : {0.3, 3.0, 40.0, 101.7, 150.0, 198.0, 204.6, 1000.0, 12345.6}) {
      const float s = (float)sig;
      const double rc = ratio * sig + 6.0 * (double)s, w = soft_width(s, rc);
      const uint32_t n = soft_bins(w, rc);
      if (n > kSoftFineMax || (n - 1) * w < rc) printf("sigma %g range %g: %u bins\n", sig, rc, n), ++bad;
      if (rc / ((double)s / 40.0) < 8180.0 && w > (double)s / 40.0) printf("sigma %g range %g: w %g\n", sig, rc, w), ++bad;
      if ((double)(float)w != w) printf("w %g\n", w), ++bad;
      for (uint32_t m = 0; m < n; ++m) {
        const double c = ((double)m + 0.5) * w;
        if ((double)(float)c != c) {
          printf("sigma %g range %g: centre of bin %u\n", sig, rc, m);
          ++bad;
          break;
        }
      }
    }
  printf(bad ? "FAIL %d\n" : "OK\n", bad);
  return bad ? 1 : 0;
}
"""


def test_fine_grid(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "fine.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "fine"
    subprocess.check_call([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "paper_2004_05188_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout
