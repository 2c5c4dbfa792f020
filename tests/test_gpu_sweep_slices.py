"""The exact path takes the pairs in slices (lo, hi] of their approximate
distance, a sweep per slice, and ends where everything below an edge has
been taken.  That needs the slices to partition the pairs: a pair's
approximate distance may not depend on the slice's edges, and a pair at or
below an edge may not be stopped by the tests that precede it.  Consecutive
slices must hold together exactly what one sweep of the whole range holds,
each pair once, with the same distance."""
import numpy as np
import pytest

from paper_2502_14446_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,d", [(1, 1), (2, 2), (3, 2), (8, 1), (8, 3), (20, 4)])
def test_slices_partition_the_pairs(D, d):
    from sweep_client import sweep
    wl = synth.tiny(70 + D, n=9001, D=D, w=64, d=d, k=3, n_motifs=2, dtype=np.float32)
    # an upper edge below which a few hundred thousand pairs lie
    hi = float(2.0 * np.sqrt(wl.w) * d)
    while True:
        hi *= 0.8
        try:
            pairs, dist = sweep(wl.series, wl.w, d, -1.0, hi, cap=1 << 19)
            break
        except AssertionError:
            continue
    assert len(pairs) > 1000
    # edges at recorded distances: a pair lies exactly on each
    edges = np.unique(np.quantile(dist, np.linspace(0.02, 0.98, 49), method="nearest").astype(np.float32))
    edges = np.concatenate([[np.float32(-1.0)], edges, [np.float32(hi)]])
    got = [sweep(wl.series, wl.w, d, float(a), float(b), cap=1 << 19) for a, b in zip(edges[:-1], edges[1:])]
    p = np.concatenate([g[0] for g in got])
    q = np.concatenate([g[1] for g in got])
    o = np.argsort(p, kind="stable")
    np.testing.assert_array_equal(p[o], pairs)
    np.testing.assert_array_equal(q[o], dist)
