"""Host check of the direct bins (r0 = 0) of the RDF over unordered pairs: with any root s within one
float32 step of sqrt(d2) (the approximate root's bound), hi, lo = (1 +- 2^-21) / dr in float32
and the clamp at (n_bins + 1/2) dr, the exact bin of d2 is floor(s hi) or, only where
floor(s lo) differs, the one below; out-of-range d2 lands in bin n_bins.  Checked on every edge
of the float32 edge table, 40 steps to both sides, and on random distances."""
import numpy as np
import pytest

f32 = np.float32


@pytest.mark.parametrize("dr,nb", [(0.01, 200), (0.02, 100), (0.003, 512), (0.001, 512), (0.1, 1), (0.05, 40),
                                   (0.0123, 163), (3.7, 511), (1e-6, 300)])
def test_bin_is_the_floor_or_the_one_below_where_the_floors_differ(dr, nb):
    E = ((np.arange(nb + 1) * np.float64(dr)) ** 2).astype(f32)
    near = [E]
    up, dn = E, E
    for _ in range(40):
        up, dn = np.nextafter(up, f32(np.inf)), np.nextafter(dn, f32(0))
        near += [up, dn]
    rng = np.random.default_rng(nb)
    d2 = np.concatenate(near + [((rng.random(200_000) * (nb + 3) * dr) ** 2).astype(f32), [f32(0)]])
    d2 = d2[(d2 == 0) | (d2 >= np.finfo(f32).tiny)]
    exact = np.searchsorted(E, d2, side="right") - 1
    hi, lo = f32((1.0 + 2.0**-21) / dr), f32((1.0 - 2.0**-21) / dr)
    far = f32((nb + 0.5) * dr)
    root = np.sqrt(d2.astype(np.float64)).astype(f32)
    for s in (root, np.nextafter(root, f32(np.inf)), np.where(d2 > 0, np.nextafter(root, f32(0)), f32(0))):
        s = np.minimum(s, far).astype(np.float64)
        m = np.floor(s * np.float64(hi)).astype(np.int64)
        same = np.floor(s * np.float64(lo)).astype(np.int64) == m
        assert np.array_equal(m[same], np.minimum(exact[same], nb))
        assert np.all((exact[~same] == m[~same]) | (exact[~same] == m[~same] - 1))
    assert (~same).mean() < 0.5
