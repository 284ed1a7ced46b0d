"""Which clouds leave the RDF of a one-pass query to the sweep over unordered pairs.  The sweep's work grows
with the records, that of the query's own pass with the centrals, so the rule has to look at
both.  Host check of the rule (include of the library's internal header, compiled for the host with
nvcc), and GPU parity with the oracle around its line."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include "ps_internal.cuh"
int main() {
  int bad = 0;
  auto is = [&](bool want, uint32_t nbr, uint32_t cells, uint32_t ctr) {
    if (ps::sweep_pays(nbr, cells, ctr) != want) printf("%u records, %u cells, %u centrals\n", nbr, cells, ctr), ++bad;
  };
  is(true, 8000000, 80000, 8000000);    // every ion about every ion
  is(true, 100000, 450, 40000);         // the ions far from the surface
  is(false, 8000000, 80000, 24000);     // solutes about every ion
  is(false, 1000000, 10000, 50000);     // the ions deep inside
  is(false, 8000000, 4000000, 8000000); // sparse clouds
  is(false, 0, 1, 0);
  is(true, 0xFFFFFFFEu, 1u << 28, 0xFFFFFFFEu);  // (no products of 32 bits)
  is(false, 0xFFFFFFFEu, 1u << 28, 1u << 28);
  printf(bad ? "FAIL %d\n" : "OK\n", bad);
  return bad ? 1 : 0;
}
"""


def test_sweep_rule(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "rule.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "rule"
    subprocess.check_call([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "paper_2004_05188_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("share", [0.0, 0.001, 0.12, 0.13, 0.14, 0.15, 1.0])
@pytest.mark.parametrize("ks", [[], [1, 10]])
def test_few_centrals_in_a_dense_cloud(orc, spec, share, ks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_2004_05188_gb300 as ps
    from test_gpu_exact import assert_same, run_gpu

    n = 6000
    xyz, _, d = spec.cube(900, n, 6.0, (1.0,))
    t = np.zeros(n, np.uint8)
    t[np.random.default_rng(3).permutation(n)[: round(share * n)]] = 1
    bins = (0.0, 0.01, 150)
    g = run_gpu(ps, xyz, t, d, [1], "all", 0.0, bins, ks, per_central=True)
    r = orc.spatstat(xyz, t, d, [1], "all", 0.0, *bins, ks, per_central=True)
    assert_same(g, r, ks, per_central=True)
