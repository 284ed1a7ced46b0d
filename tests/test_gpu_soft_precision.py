"""The smoothed RDF keeps what float32 distances hold, also where a few equal pairs make up the sums.

Blocks of m^3 ions on 64 lattice constants, h against FP64 over all pairs.  Scale of the error, the sum over the
pairs of its largest parts: float32 distance |K'| u 2^-22 (three roundings of the squared distance, the
root's bound of 2^-23), the expansion's third order |K'''| (w / 2)^3 / 6 with w = sigma / 40, and the
rounding of the result 2^-24 |h|.  Each is far below its largest on average: a remainder that is uniform in a
bin has a cube of 1 / sqrt(7) = 0.38 of the largest in the quadratic mean, a sum of several roundings
less.  So the quadratic mean over the lattices has to stay below 0.38 of that scale."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _derivatives(e, u, s):
    from math import erf

    t = (e[:, None] - u[None, :]) / s
    ph = np.exp(-0.5 * t * t) / np.sqrt(2.0 * np.pi)
    k0 = 0.5 * (1.0 + np.vectorize(erf)(t / np.sqrt(2.0)))
    return [np.diff(k, axis=0) for k in (k0, -ph / s, (1.0 - t * t) * ph / s**3)]


@pytest.mark.parametrize("sig,stop,nb,m", [(0.2, 0.3, 6, 2), (2.0, 2.0, 20, 2), (0.5, 0.4, 8, 2), (0.05, 0.3, 6, 2),
                                           (0.05, 2.0, 100, 3), (1.0, 2.0, 20, 4)])
def test_remainders_of_equal_pairs(sig, stop, nb, m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_2004_05188_gb300 as ps

    bins, rc, e = (0.0, stop / nb, nb), stop + 6.0 * sig, np.arange(nb + 1) * (stop / nb)
    rel = []
    for a in np.linspace(0.2, 0.42, 64):
        k = np.arange(m) * a
        x = np.stack(np.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3).astype(np.float32)
        i, j = np.triu_indices(len(x), 1)
        u = np.linalg.norm(x[j].astype(np.float64) - x[i], axis=1)
        u = u[u < rc]
        k0, k1, k3 = (2.0 * v for v in _derivatives(e, u, sig))
        ref = k0.sum(1)
        scale = (np.abs(k1) * u).sum(1) * 2.0**-22 + np.abs(k3).sum(1) * (sig / 80.0) ** 3 / 6.0 + 2.0**-24 * np.abs(ref)
        X = torch.from_numpy(x).cuda()
        T = torch.zeros(len(x), dtype=torch.uint8, device="cuda")
        g = ps.Grid(len(x)).build(X, T, "all", ps.soft_r_cut(bins, sig, 1.0))
        h = ps.soft_rdf_fwd(g, None, "all", 0.0, sig, 1.0, bins).cpu().numpy().astype(np.float64)
        rel.append(np.linalg.norm(h - ref) / np.linalg.norm(scale))
        g.close()
    assert np.sqrt(np.mean(np.square(rel))) < 0.38
