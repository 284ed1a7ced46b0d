"""A histogram range whose square underflows float32: no neighbour is in range, and the in-range counts are 0."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,L", [(3000, 4.0), (300, 6.0)])
@pytest.mark.parametrize("dr", [1e-30, 1e-22, 1e-12])
@pytest.mark.parametrize("rdf", [True, False])
def test_counts_of_a_vanishing_range(spec, n, L, dr, rdf):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_2004_05188_gb300 as ps
    from test_gpu_exact import run_gpu

    xyz, t, d = spec.cube(800 + n, n, L, (0.5, 0.5))
    for ctr, nbr in (("all", "all"), ([0], [1]), ([0], [0, 1])):
        g = run_gpu(ps, xyz, t, d, ctr, nbr, 0.0, (0.0, dr, 3), [1, 3], per_central=True, r_cut=1.0, rdf=rdf)
        central = np.ones(n, bool) if ctr == "all" else t == 0
        np.testing.assert_array_equal(g["n_within"][central], 0)
        assert g["meta"][0] == central.sum() and g["meta"][3] == 0
        np.testing.assert_array_equal(g["meta"][4::2], central.sum())  # no k-th neighbour found
        assert not g["knn"].any() and not (rdf and g["rdf"].any())
