"""Forces of the smoothed RDF on a lattice, where they cancel, and queries whose central work lists are made
inside the scan of the cell counts (grids of 2^18 and more cells, centrals not among the neighbours)."""
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


@pytest.mark.parametrize("cs", [1.0, 0.5])
@pytest.mark.parametrize("copies", [1, 6])
def test_lattice_forces_cancel(ps, spec, cs, copies):
    """Ions further than the range from the faces of a simple-cubic block of coincident copies: each force
    f meets its opposite, so what is left is float32's rounding of a sum of n_pair terms, below
    n_pair 2^-23 times the sum of their sizes (both ends of a pair act: twice).  The forces of the whole
    block add up to zero likewise."""
    m, a, sig, bins = 16, 0.25, 0.05, (0.0, 0.02, 30)
    rc = bins[1] * bins[2] + 6 * sig
    xyz, t, d = spec.simple_cubic(m, a, 0.125)
    xyz, t, d = (np.repeat(v, copies, axis=0) for v in (xyz, t, d))
    X, T, D = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (xyz, t, d))
    g = ps.Grid(X.shape[0], cs).build(X, T, "all", ps.soft_r_cut(bins, sig, 1.0))
    G = np.random.default_rng(7).normal(size=bins[2]).astype(np.float32)
    gx, _ = ps.soft_rdf_bwd(g, D, "all", -1.0, sig, 1.0, bins, torch.from_numpy(G).cuda())
    gx = gx.cpu().numpy().astype(np.float64)
    k = np.arange(-4, 5)
    u = a * np.sqrt(sum(v**2 for v in np.meshgrid(k, k, k, indexing="ij")).ravel())
    u = u[(u < rc) & (u > 0)]
    e = np.arange(bins[2] + 1) * bins[1]
    pdf = np.exp(-0.5 * ((e[None, :] - u[:, None]) / sig) ** 2) / sig / np.sqrt(2 * np.pi)
    size = 2.0 * copies * np.abs(-(np.diff(pdf, axis=1) * G).sum(1)).sum()
    n_pair = copies * len(u)
    lo, hi = xyz.min(0) + rc, xyz.max(0) - rc
    inside = np.all((xyz > lo) & (xyz < hi), axis=1)
    assert inside.sum() >= 100 * copies
    assert np.abs(gx[inside]).max() <= n_pair * 2.0**-23 * size
    assert np.abs(gx).max() > 1e-3 * size  # the ions at the faces do feel a force
    assert np.abs(gx.sum(0)).max() <= n_pair * 2.0**-23 * size * np.sqrt(len(gx))
    g.close()


@pytest.mark.parametrize("ks,per", [([1, 6], True), ([], False)])
def test_work_lists_made_in_the_scan(ps, orc, spec, ks, per):
    n, L, bins = 300_000, 32.3, (0.0, 0.01, 100)
    xyz, t, d = spec.cube(99, n, L, (0.3, 0.7))
    X, T, D = (torch.from_numpy(v).cuda() for v in (xyz, t, d))
    g = ps.Grid(n, 0.5).build(X, T, "all", 1.0 + 1e-6)
    assert g.info()["n_cells"] >= 1 << 18
    from test_gpu_exact import assert_same

    for ctr, nbr in (([0], [1]), ([0, 1], [1])):
        g.build(X, T, nbr, 1.0 + 1e-6)
        assert g.info()["n_cells"] >= 1 << 18
        out = ps.spatstat(g, D, ctr, 0.3, bins, ks, per_central=per)
        res = {k: (v.cpu().numpy() if v is not None else None) for k, v in out.items()}
        r = orc.spatstat(xyz, t, d, ctr, nbr, 0.3, *bins, ks, per_central=per)
        assert_same(res, r, ks, per_central=per)
    g.close()
