"""GPU parity of the distribution map with the oracle where few of the neighbour records are central (a warp
per central instead of the sweep over unordered pairs), around the rule's line, on dense and thin
clouds and all stencils; and the rule itself."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ps():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_2004_05188_gb300 as ps

    return ps


@pytest.mark.parametrize("n,L", [(5000, 5.0), (5000, 20.0), (700, 2.0), (40, 0.5)])
@pytest.mark.parametrize("cs", [1.0, 0.5, 1 / 3])
@pytest.mark.parametrize("nv,w", [(30, 0.1), (31, 0.1), (7, 0.25)])
def test_map_of_few_centrals(ps, orc, spec, n, L, cs, nv, w):
    R = 1.4
    xyz, _, d = spec.cube(500 + n, n, L, (1.0,))
    xyz, d = np.concatenate([xyz, xyz[:9]]), np.concatenate([d, d[:9]])
    order = np.random.default_rng(n).permutation(len(xyz))
    g = ps.Grid(len(xyz), cs)
    X, D = torch.from_numpy(np.ascontiguousarray(xyz)).cuda(), torch.from_numpy(d).cuda()
    for few in (0, 1, 5, len(xyz) // 40, len(xyz) // 25, len(xyz) // 8, len(xyz)):
        t = np.zeros(len(xyz), np.uint8)
        t[order[:few]] = 3
        g.build(X, torch.from_numpy(t).cuda(), "all", R * (1 + 1e-6))
        out = ps.sdm(g, D, [3], 0.0, R, w, nv)
        H, m = orc.sdm(xyz, t, d, [3], "all", 0.0, R, w, nv)
        np.testing.assert_array_equal(out["meta"].cpu().numpy()[:3].astype(np.uint64), m)
        np.testing.assert_array_equal(out["H"].cpu().numpy().astype(np.uint64), H)
    g.close()
