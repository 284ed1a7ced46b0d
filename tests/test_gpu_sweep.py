"""GPU parity of the sweep over unordered pairs (the RDF of the query in passes) against the oracle,
at the sizes where it can go wrong: blocks of 1 .. 200 records (partly filled tiles, several staged
groups), central and other records mixed in a block, the direct bins at their limit (512 bins) and
the general ones beside it (513 bins, r0 > 0), pairs exactly on the edges, coincident ions, and
clouds of few cells whose candidates are split into parts."""
import numpy as np
import pytest

from test_gpu_exact import assert_same, run_gpu

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


@pytest.mark.parametrize("n,L,cs", [(2, 0.5, 0.5), (63, 1.0, 0.5), (64, 1.0, 0.75), (65, 1.0, 0.5), (700, 2.0, 0.75),
                                    (3000, 12.0, 1 / 3), (9000, 9.0, 0.4), (5000, 40.0, 0.5)])
@pytest.mark.parametrize("bins", [(0.0, 0.005, 300), (0.0, 1.5 / 512, 512), (0.0, 1.5 / 513, 513), (0.4, 0.1, 11),
                                  (0.0, 1.5, 1)])
def test_rdf_over_unordered_pairs(ps, orc, spec, n, L, cs, bins):
    xyz, t, d = spec.cube(300 + n, n, L, (0.5, 0.5))
    half = float(np.median(d))  # about half of the ions central
    for ctr, nbr, dmin in (("all", "all", -1.0), ("all", "all", half), ([1], "all", 0.0)):
        g = run_gpu(ps, xyz, t, d, ctr, nbr, dmin, bins, [], cell_scale=cs, split=True)
        r = orc.spatstat(xyz, t, d, ctr, nbr, dmin, *bins, [])
        assert_same(g, r, [])


def test_lattice_edges_and_coincident_ions(ps, orc, spec):
    xyz, t, d = spec.simple_cubic(14, 0.25, 0.125)  # every distance on or near an edge
    xyz = np.concatenate([xyz, xyz[:100], xyz[:7]])
    t, d = np.zeros(xyz.shape[0], np.uint8), np.concatenate([d, d[:100], d[:7]])
    for bins in ((0.0, 0.01, 150), (0.0, 0.25, 6), (0.25, 0.25, 5)):
        for dmin in (0.0, 0.6):
            g = run_gpu(ps, xyz, t, d, "all", "all", dmin, bins, [], cell_scale=0.5, split=True)
            r = orc.spatstat(xyz, t, d, "all", "all", dmin, *bins, [])
            assert_same(g, r, [])


@pytest.mark.parametrize("R,w,nv", [(1.5, 0.1, 30), (1.5, 0.1, 31), (1.0, 0.25, 8), (1.0, 0.25, 7), (1.2, 3.0, 1)])
@pytest.mark.parametrize("lattice", [False, True])
def test_distribution_map_mirrored(ps, orc, spec, R, w, nv, lattice):
    """The map from unordered pairs: mirrored voxels, odd cubes (a voxel that is its own mirror
    image), displacements on voxel edges, one or both ends central, coincident ions."""
    if lattice:
        xyz, t, d = spec.simple_cubic(11, 0.25, 0.125)
    else:
        xyz, t, d = spec.cube(77, 1500, 4.0, (0.5, 0.5))
    xyz, t, d = np.concatenate([xyz, xyz[:20]]), np.concatenate([t, t[:20]]), np.concatenate([d, d[:20]])
    X, T, D = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (xyz, t, d))
    for cs, dmin, ctr in ((1.0, 0.5, "all"), (0.5, 0.3, [0])):
        g = ps.Grid(X.shape[0], cs).build(X, T, "all", R * (1 + 1e-6))
        out = ps.sdm(g, D, ctr, dmin, R, w, nv)
        H, m = orc.sdm(xyz, t, d, ctr, "all", dmin, R, w, nv)
        np.testing.assert_array_equal(out["meta"].cpu().numpy()[:3].astype(np.uint64), m)
        np.testing.assert_array_equal(out["H"].cpu().numpy().astype(np.uint64), H)
        g.close()


@pytest.mark.parametrize("m,copies", [(12, 1), (12, 3), (24, 40)])
def test_smoothed_rdf_of_lattice_shells(ps, spec, m, copies):
    """Smoothed RDF and dL/dscale of coincident copies of a simple-cubic block against the closed form
    over its shells (FP64): every pair of a shell falls into one fine bin, up to 2e8 of them (the
    integer moments are drained on the way), and coincident ions count at u = 0 but the ion itself
    does not.  Tolerance: the library's stated 1e-5 of h; the force of each interior ion cancels."""
    from math import erf, exp, pi, sqrt

    a, sig, bins = 0.25, 0.05, (0.0, 0.02, 30)
    xyz, t, d = spec.simple_cubic(m, a, 0.125)
    xyz, t, d = (np.repeat(v, copies, axis=0) for v in (xyz, t, d))
    rc = 0.6 + 6 * sig
    dmin = 0.95
    X, T, D = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (xyz, t, d))
    g = ps.Grid(X.shape[0], 0.5).build(X, T, "all", ps.soft_r_cut(bins, sig, 1.0))
    h = ps.soft_rdf_fwd(g, D, "all", dmin, sig, 1.0, bins).cpu().numpy().astype(np.float64)
    G = np.random.default_rng(5).normal(size=bins[2])
    gx, gs = ps.soft_rdf_bwd(g, D, "all", dmin, sig, 1.0, bins, torch.from_numpy(G.astype(np.float32)).cuda())
    n_c = int((d >= dmin).sum())
    assert n_c > 0
    k = np.arange(-4, 5)
    I, J, K = np.meshgrid(k, k, k, indexing="ij")
    u = a * np.sqrt((I**2 + J**2 + K**2).ravel())
    u = u[u < rc]
    e = np.arange(bins[2] + 1) * bins[1]
    Phi = np.array([[0.5 * (1 + erf((x - y) / sig / sqrt(2))) for x in e] for y in u])
    pdf = np.array([[exp(-0.5 * ((x - y) / sig) ** 2) / sig / sqrt(2 * pi) for x in e] for y in u])
    mult = np.where(u > 0, copies, copies - 1).astype(np.float64)
    ref = n_c * (mult[:, None] * np.diff(Phi, axis=1)).sum(0)
    assert np.linalg.norm(h - ref) <= 1e-5 * np.linalg.norm(ref)
    W = -(np.diff(pdf, axis=1) * G.astype(np.float32)).sum(1)
    gs_ref = n_c * (mult * W * u).sum()
    assert abs(float(gs[0]) - gs_ref) <= 1e-4 * n_c * (mult * np.abs(W) * u).sum()
    g.close()


@pytest.mark.parametrize("n,L", [(40, 9.0), (900, 9.0), (5000, 9.0), (12000, 7.0), (9000, 3.5), (30, 1.0)])
@pytest.mark.parametrize("bins", [(0.0, 0.01, 200), (0.3, 0.05, 34)])
def test_default_grid_over_its_densities(ps, orc, spec, n, L, bins):
    """Default options from a record per cell to hundreds (RDF and in-range counts in the query or in
    the sweep, cells without sub-cells, with 8 and with 64), centrals among the neighbours or not,
    one to sixteen lanes per central, a blob that fills single cells."""
    xyz, t, d = spec.cube(400 + n, n, L, (0.5, 0.3, 0.2))
    blob = (np.array([L / 3, L / 2, L / 2]) + np.random.default_rng(n).normal(0, 0.05, (n // 10, 3))).astype(np.float32)
    xyz = np.concatenate([xyz, blob, xyz[:3]])
    t, d = np.resize(t, xyz.shape[0]), np.resize(d, xyz.shape[0])
    for ctr, nbr, dmin, ks in (("all", "all", 0.0, [1, 3, 32]), ([0], [0, 1], 0.4, [10]), ([0, 2], [1], 0.0, [2, 5]),
                               ("all", "all", 0.6, [])):
        g = run_gpu(ps, xyz, t, d, ctr, nbr, dmin, bins, ks, per_central=True)
        r = orc.spatstat(xyz, t, d, ctr, nbr, dmin, *bins, ks, per_central=True)
        assert_same(g, r, ks, per_central=True)


@pytest.mark.parametrize("n,L", [(3, 1.0), (40, 3.0), (2500, 5.0), (6000, 12.0)])
@pytest.mark.parametrize("cs", [1.0, 0.5])
@pytest.mark.parametrize("k", [1, 10, 13, 16, 17, 32])
def test_knn_and_counts_without_the_rdf(ps, orc, spec, n, L, cs, k):
    """k-th distances and in-range counts alone (both from one distance, near and far candidates),
    one to sixteen lanes per central, the bound over the lanes of a central for the longer lists."""
    xyz, t, d = spec.cube(700 + n, n, L, (0.5, 0.5))
    xyz = np.concatenate([xyz, xyz[:2]])
    t, d = np.resize(t, xyz.shape[0]), np.resize(d, xyz.shape[0])
    bins = (0.0, 0.02, 75)
    for ctr, nbr in (("all", "all"), ([0], [1])):
        for per_central in (True, False):
            g = run_gpu(ps, xyz, t, d, ctr, nbr, 0.0, bins, [1, k], per_central=per_central, cell_scale=cs, rdf=False)
            r = orc.spatstat(xyz, t, d, ctr, nbr, 0.0, *bins, [1, k], per_central=per_central)
            assert_same(g, r, [1, k], per_central=per_central, rdf=False)
