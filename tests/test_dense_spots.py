"""Clouds with a very dense spot, where single blocks of the sweep over unordered pairs hold more work than a
warp's share: the rule that lists their records in groups (host check, include of the library's
internal header compiled with nvcc), and GPU parity with the oracle where groups are listed."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include "ps_internal.cuh"
using namespace ps;
int main() {
  int bad = 0;
  const uint32_t warps = 152 * 32;
  auto is = [&](bool want, const char* what, uint32_t n, uint32_t n_cand, uint32_t n_sel, uint32_t n_cells, int st) {
    const uint32_t S = sweep_parts(n_cells / sweep_block(n_cells, n_sel), warps);
    if (heavy_block(n, n_cand, n_sel, n_cells, S, warps, st) != want) printf("%s\n", what), ++bad;
  };
  // even clouds, the fullest blocks
  is(false, "needle 8e6, 2 nm", 300, 27 * 260, 8000000, 77000, 1);
  is(false, "needle 8e6, 1 nm", 50, 125 * 35, 8000000, 600000, 2);
  is(false, "needle 1e6, 2 nm", 300, 27 * 260, 1000000, 10400, 1);
  is(false, "cylinder 1e5, 2 nm", 400, 27 * 340, 100000, 450, 1);
  is(false, "cylinder 2e4, 2 nm", 400, 27 * 340, 20000, 290, 1);
  // dense spots
  is(true, "5e4 ions in a few cells of 2e6", 5000, 50000, 2050000, 67000, 2);
  is(true, "a cell at the edge of that spot", 200, 40000, 2050000, 67000, 2);
  is(true, "2e5 ions in 8 cells", 25000, 200000, 200000, 8, 1);
  // the groups of the listed blocks fit their array
  for (uint64_t n = kHeavyGroup + 1; n < 4000; ++n)
    for (uint64_t blocks = 1; blocks < 2000; blocks += 37)
      if (blocks * ((n + kHeavyGroup - 1) / kHeavyGroup) > heavy_capacity(blocks * n)) ++bad;
  printf(bad ? "FAIL %d\n" : "OK\n", bad);
  return bad ? 1 : 0;
}
"""


def test_heavy_blocks(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    src = tmp_path / "heavy.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "heavy"
    subprocess.check_call([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "paper_2004_05188_gb300", "csrc"),
                           "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout


def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_2004_05188_gb300 as ps

    return ps, torch


def _cloud(n, L, blob, sig, seed):
    rng = np.random.default_rng(seed)
    x = np.concatenate([rng.random((n, 3)) * L, L / 3 + sig * rng.standard_normal((blob, 3))]).astype(np.float32)
    x = np.concatenate([x, x[:5], x[-5:]])  # coincident ions in both
    return x, rng.integers(0, 3, len(x)).astype(np.uint8), rng.random(len(x)).astype(np.float32)


@pytest.mark.gpu
@pytest.mark.parametrize("n,L,blob,sig", [(6000, 7.0, 4001, 0.2), (300, 1.0, 6000, 0.1), (20000, 14.0, 3000, 0.02),
                                          (0, 1.0, 5000, 0.4)])
@pytest.mark.parametrize("cs,split", [(1.0, False), (0.5, False), (0.5, True), (1 / 3, True)])
def test_query_with_a_dense_spot(orc, n, L, blob, sig, cs, split):
    ps, _ = _gpu()
    from test_gpu_exact import assert_same, run_gpu

    xyz, t, d = _cloud(n, L, blob, sig, 40 + blob)
    for ctr, dmin, bins in (("all", 0.0, (0.0, 0.01, 120)), ([1, 2], 0.5, (0.0, 0.01, 120)), ("all", 0.0, (0.2, 0.1, 10))):
        per = not split
        g = run_gpu(ps, xyz, t, d, ctr, "all", dmin, bins, [1, 7], per_central=per, cell_scale=cs, split=split)
        r = orc.spatstat(xyz, t, d, ctr, "all", dmin, *bins, [1, 7], per_central=per)
        assert_same(g, r, [1, 7], per_central=per)


@pytest.mark.gpu
@pytest.mark.parametrize("cs", [1.0, 0.5])
def test_several_statistics_of_one_build(orc, cs):
    """One build, first a query that leaves the sweep out (the groups are not listed), then ones that use it
    twice (listed once), the distribution map, and the smoothed RDF with its adjoint."""
    ps, torch = _gpu()
    xyz, t, d = _cloud(2500, 9.0, 1500, 0.15, 9)
    X, T, D = (torch.from_numpy(a).cuda() for a in (xyz, t, d))
    bins, sig, sb = (0.0, 0.01, 100), 0.05, (0.0, 0.02, 50)
    g = ps.Grid(X.shape[0], cs).build(X, T, "all", ps.soft_r_cut(sb, sig, 1.0))
    for ctr, dmin in (([0], 0.97), ("all", 0.0), ("all", 0.3)):
        o = ps.spatstat(g, D, ctr, dmin, bins, [2])
        r = orc.spatstat(xyz, t, d, ctr, "all", dmin, *bins, [2])
        np.testing.assert_array_equal(o["rdf"].cpu().numpy().astype(np.uint64), r["rdf"])
        np.testing.assert_array_equal(o["knn"].cpu().numpy().astype(np.uint64), r["knn"])
    for ctr in ("all", [2]):
        o = ps.sdm(g, D, ctr, 0.0, 1.0, 0.1, 20)
        H, m = orc.sdm(xyz, t, d, ctr, "all", 0.0, 1.0, 0.1, 20)
        np.testing.assert_array_equal(o["H"].cpu().numpy().astype(np.uint64), H)
    G = np.random.default_rng(1).standard_normal(sb[2])
    h = ps.soft_rdf_fwd(g, D, "all", 0.0, sig, 1.0, sb).cpu().numpy().astype(np.float64)
    gx, gs = ps.soft_rdf_bwd(g, D, "all", 0.0, sig, 1.0, sb, torch.from_numpy(G.astype(np.float32)).cuda())
    href = orc.soft_fwd(xyz, t, d, "all", "all", 0.0, sig, 1.0, *sb)
    gref, gsref = orc.soft_bwd(xyz, t, d, "all", "all", 0.0, sig, 1.0, *sb, G)
    assert np.linalg.norm(h - href) <= 1e-5 * np.linalg.norm(href)
    assert np.linalg.norm(gx.cpu().numpy() - gref) <= 1e-4 * np.linalg.norm(gref)
    assert abs(float(gs[0]) - gsref) <= 1e-4 * abs(gsref)
    g.close()
