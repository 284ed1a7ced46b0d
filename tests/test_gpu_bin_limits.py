"""Queries in passes whose kNN histograms nearly fill the shared memory are accepted, whichever kernel does the
near pass."""
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


@pytest.mark.parametrize("nb", [1417, 1418, 1419, 1430, 1440])
@pytest.mark.parametrize("ks", [list(range(1, 33)), [10] * 32])
def test_most_bins_in_passes(ps, orc, spec, nb, ks):
    from test_gpu_exact import assert_same, run_gpu

    xyz, t, d = spec.cube(60 + nb, 3000, 5.0, (0.6, 0.4))
    bins = (0.0, 0.001, nb)
    r = orc.spatstat(xyz, t, d, "all", "all", 0.4, *bins, ks)
    for cs in (0.5, 1 / 3):
        g = run_gpu(ps, xyz, t, d, "all", "all", 0.4, bins, ks, cell_scale=cs, split=True)
        assert_same(g, r, ks)
